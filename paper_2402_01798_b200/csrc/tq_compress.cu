// Client side of Algorithm 1: truncate (Section 3.1, truncation equation), stochastically round onto
// the codebook (Section 3.1, quantizer equation) and pack b-bit codes, fused in one pass.
//
// Work split: a thread owns a run of 32 consecutive elements = four groups of 8, a tile is one run for each of a block's 256
// threads.  A group is the unit of randomness: one Philox4x32-10 call (counter = group index, worker) yields 128
// bits = eight 16-bit slots, one per element.  A run packs into exactly `bits` 32-bit words, so no thread ever shares a
// word with another and no shuffles or atomics are needed.
//   Quantizers in kernel parameters (compress_kernel): a grid row per worker, the lookup tables built before the data is
//   waited for; blocks of table codebooks and of bf16 rows take several tiles.
//   Quantizers in device memory (compress_kernel_dev): the tiles of all jobs cut into contiguous ranges (TilePlan).
// HBM traffic per element: 4 (fp32) or 2 (bf16) bytes read, bits/8 bytes written.
//
// What bounds it: fp32 rows come close to HBM (25.6 M x 16, 16 levels: 327 us, 282 at the rate of a plain copy; 4 levels
// 30 M x 8: 150 us, 156), bf16 rows the multiplier pipe, which Philox's wide multiplies occupy for 9 cycles per 32
// elements.  So the per-element arithmetic runs on the multiply-add pipes or on the integer / compare pipe,
// whichever has room, where the result is provably the same:
//   - floor / int conversion: add 2^23 rounding down, the integer appears in the mantissa;
//   - threshold T = rint(p * 2^16): one fused multiply-add with 2^23;
//   - interval and threshold together as the one integer X = k * 2^16 + T, code = floor((X + 65535 - r) / 2^16); for the uniform codebook
//     X = rint(x * 2^16) at once, with the clamps of x done by saturating multiplies and a minimum;
//   - codes are packed by byte-permutes and products of integers;
//   - (binary search and the unscaled uniform form only) the random slot r as the float 2^23 + r: one byte-permute; [r < T] =
//     sat((2^23 + T) - (2^23 + r)), a saturating subtract of two exactly representable integers;
//   - table offsets are formed as denormal floats whose bit pattern IS the byte offset.
#include <cmath>
#include <cstring>

#include "tq_device.cuh"
#include "tq_launch.h"
#include "tq_lut.cuh"

namespace tq {

constexpr int kMaxGridCells = 2048;   // finest lookup grid for the non-uniform interval search
constexpr int kMinGridCells = 32;

// Per-worker quantizer as the kernel sees it.
struct WorkerQ {
    float alpha, inv_step, top;   // top = (float)(L-1)
    float inv_step_l;             // inv_step / L when that quotient is exact and normal, else 0 (uniform mode)
    float inv_2alpha;             // maps [-alpha, alpha] to [0, 1] for the lookup grid
    float cell_scale;             // grid cells M as the denormal M * 2^-149
    uint32_t cells;               // M, 0: no linear grid separates the levels
    uint32_t log_base, log_cells; // logarithmic grid: 8 * first cell, cells per sign (0: it does not separate them either)
    float levels[TQ_MAX_LEVELS];
    float inv_width[TQ_MAX_LEVELS];
};
// By-value arguments are copied at every launch: calls of few workers do not pass room for all.
constexpr uint32_t kFewWorkers = 16;
template <uint32_t N>
struct CompressArgs {
    WorkerQ q[N];
};

// kUniformWide: the uniform codebook through the arithmetic that needs no scaled inverse step (used
// only when inv_step / L would be subnormal, i.e. alpha beyond about 2^121).
enum Search { kUniform = 0, kGrid = 1, kBinary = 2, kUniformWide = 3, kLogGrid = 4 };
__host__ __device__ constexpr bool is_uniform(int search) { return search == kUniform || search == kUniformWide; }

cudaError_t launch_compress_dev(const CompressCall& c);

__device__ __forceinline__ float mul_sat(float a, float b) {
    float r; asm("mul.rn.sat.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r;
}
__device__ __forceinline__ float sub_sat(float a, float b) {
    float r; asm("sub.rn.sat.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r;
}
__device__ __forceinline__ float set_ge(float a, float b) {   // 1.0f if a >= b else 0.0f (0 for NaN)
    float r; asm("set.ge.f32.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r;
}

// Grid cell of a value: floor(M * sat((g + alpha) * inv_2alpha)), returned as a float whose BIT
// PATTERN is that integer (a denormal).  Monotone in g; NaN maps to cell 0.  The same expression is
// evaluated on the host (cell_of below) when the grid resolution is chosen.
__device__ __forceinline__ float grid_cell(float g, float alpha, float inv_2alpha, float cell_scale) {
    return __fmul_rd(mul_sat(__fadd_rn(g, alpha), inv_2alpha), cell_scale);
}

// [r < T] as 1.0f / 0.0f, where T = rint(p * 2^16) and rf = 2^23 + r.  Both operands of the subtract
// are integers below 2^24, so the difference is exact; huge or infinite p saturate correctly and a
// NaN gives 0.
__device__ __forceinline__ float rounds_up(float p, float rf) {
    return sub_sat(__fmaf_rn(p, 65536.0f, kMagic), rf);
}

// Uniform codebook, l_k = -alpha + k * 2 alpha / s (Section 4.1), two elements at a time.  Reference
// form of the decision: t = clip(g), x = (t + alpha) * inv_step, k = min(floor x, s-1), p = x - k,
// T = rint(p * 2^16), code = k + [r < T].
//
// Computed here through the single integer X = rint(x * 2^16): since k * 2^16 is an integer,
// X = k * 2^16 + T (a carry when T = 2^16 is the next interval with T = 0, the same code), and
// code = k + [r < T] = ceil((X - r) / 2^16) for 0 <= r < 2^16.  With L = s + 1 a power of two:
//   sum = g + alpha                            (as the reference; for |g| <= alpha it is t + alpha)
//   y   = sat(sum * (inv_step / L))            = clip(x, 0, L) / L exactly: scaling by a power of two commutes
//                                                with the rounding of the product, and .sat sends NaN and
//                                                negatives to 0, which is where the reference sends them
//   y   = min(y, s/L)                          this is x = s, which the reference codes as s, like every g >= alpha
//   Xm  = fma(y, L * 2^16, 2^23)               = 2^23 + X, rounded to nearest-even as rint does (2^23 is even)
//   v   = bits(Xm) - r + 65535                 = 0x4B000000 + (X - r + 65535): the code is byte 2 of v
// From Xm on integers do the work.  fp32 rows: a mask or shift and one three-operand addition of the integer / compare pipe (30 M x 8,
// 4 levels 150 us, 156 at a copy's rate).  bf16 rows are bound by the multiplier pipe, which Philox's wide multiplies keep busy for 9
// cycles per 32 elements, and the integer pipe (2 per logic operation or byte permute): there the complement of a word of random bits,
// 65535 - r in either half, goes through a two-way dot product (124 M x 8, 4 / 8 / 16 levels, device parameters for 4 and 8: 489 / 515 / 485
// us; slots as floats by byte permutes, then packed subtractions and multiplications of denormals: 528 / - / 510; as for fp32: 8 levels 560.
// For fp32 rows it is the slower form: 25.6 M x 16, 16 levels 265 -> 270).
// sum0 / sum1 are g + alpha of the pair.
struct UniformQ {
    float inv_step_l, c_top;      // inv_step / L, s / L
    f32x2 scale2;                 // L * 2^16, twice
};
// min(y, s/L) runs on the integer/compare pipe as well.
template <bool BF16>
__device__ __forceinline__ void code_uniform2(float sum0, float sum1, const UniformQ& u, uint32_t rnd, uint32_t& v0, uint32_t& v1) {
    float x0, x1;
    unpair(fma2(pair(fminf(mul_sat(sum0, u.inv_step_l), u.c_top), fminf(mul_sat(sum1, u.inv_step_l), u.c_top)), u.scale2, both(kMagic)), x0, x1);
    if constexpr (BF16) {
        v0 = dot_halves(~rnd, 0x0001u, __float_as_uint(x0));
        v1 = dot_halves(~rnd, 0x0100u, __float_as_uint(x1));
    } else {
        v0 = __float_as_uint(x0) - (rnd & 0xFFFFu) + 0xFFFFu;
        v1 = __float_as_uint(x1) - (rnd >> 16) + 0xFFFFu;
    }
}

// The same decision without the scaled inverse step (alpha so large that inv_step / L is subnormal):
// x = clip((g + alpha) * inv_step, 0, s), k' = floor x, p' = x - k'; at x = s this yields k' = s, p' = 0,
// i.e. the same code s as k = s-1, p >= 1.  NaN becomes 0 (fmaxf drops it).  Returns the plain code.
__device__ __forceinline__ f32x2 code_uniform2_wide(float sum0, float sum1, f32x2 inv_step2, float top, float rf0, float rf1) {
    float x0, x1;
    unpair(mul2(pair(sum0, sum1), inv_step2), x0, x1);
    const f32x2 x = pair(fminf(fmaxf(x0, 0.0f), top), fminf(fmaxf(x1, 0.0f), top));
    const f32x2 magic2 = both(kMagic);
    const f32x2 kf = sub2(add2_rd(x, magic2), magic2);                       // floor(x), exact
    float pm0, pm1;
    unpair(fma2(sub2(x, kf), both(65536.0f), magic2), pm0, pm1);            // 2^23 + rint(p * 2^16)
    return add2(kf, pair(sub_sat(pm0, rf0), sub_sat(pm1, rf1)));
}

// g + alpha for elements 2h and 2h+1 of a loaded group.  bf16 storage: the widening is part of the add
// (the stored 16 bits are an exact fp32 value, so the sum rounds as the fp32 add of the widened value).
template <bool BF16>
__device__ __forceinline__ void pair_plus_alpha(const Raw8<BF16>& g, int h, float alpha, float& sum0, float& sum1) {
    if constexpr (BF16) {
        asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %2;\n\tadd.rn.f32.bf16 %0, lo, %3;\n\tadd.rn.f32.bf16 %1, hi, %3;\n\t}"
            : "=f"(sum0), "=f"(sum1) : "r"(g.v[h]), "f"(alpha));
    } else {
        unpair(add2(pair(__uint_as_float(g.v[2 * h]), __uint_as_float(g.v[2 * h + 1])), both(alpha)), sum0, sum1);
    }
}

// General codebook through the lookup grid, two elements at a time.  s_grid[c] = (boundary, 8 k_lo): k_lo
// counts the interior levels in cells below c and `boundary` is the one interior level inside cell c
// (NaN if none, so that not even +inf compares >= it), so
// k = k_lo + [g >= boundary] = max{ j <= s-1 : l_j <= g }.  s_cell[k] = (l_k, 1/|Delta_k|).
// g is not clipped first: beyond +-alpha the same interval is found as for the clipped value, and
// p >= 1 (or p < 0, or NaN) saturates to the same decision.
// What follows an 8-byte lookup is scalar: to use the two halves of two lookups as pairs takes a move per value, which
// costs an issue slot and often the multiplier pipe, more than pairing saves (25.6 M x 16, 16 levels: 355 -> 349 us, through
// device parameters 394 -> 350 us; 250 M x 4, 8 levels 958 -> 861 us).
// The kernel is near HBM's rate with issue, multiplier, shared-memory and integer pipes all at 60-80 %, and at the GPU's power limit in
// long runs, so every operation counts.  k appears only as the denormal 8k * 2^-149, whose bit pattern is the byte offset into s_cell and,
// shifted, k * 2^16; T as the mantissa of 2^23 + T with p saturated by its product (T stays within 0 .. 2^16, 0 for a NaN); the
// sum of the two and 65535 - r, from the complement of the random word, by a two-way dot product has the code in byte 2.  With k, [r < T] and the code as
// floats: 25.6 M x 16, 16 levels, host / device parameters 329 / 335 us, now 310 / 322; 250 M x 4, 8 levels 796, now 779; 1 M x 8 12.0, 11.5.
__device__ __forceinline__ void code_cells2(float g0, float g1, float2 gc0, float2 gc1, const char* s_cell, uint32_t rnd, uint32_t& v0, uint32_t& v1) {
    const float eight = __uint_as_float(8u);
    const uint32_t k0 = __float_as_uint(__fmaf_rn(set_ge(g0, gc0.x), eight, gc0.y)), k1 = __float_as_uint(__fmaf_rn(set_ge(g1, gc1.x), eight, gc1.y));
    const float2 q0 = *reinterpret_cast<const float2*>(s_cell + k0);
    const float2 q1 = *reinterpret_cast<const float2*>(s_cell + k1);
    const float p0 = mul_sat(__fsub_rn(g0, q0.x), q0.y), p1 = mul_sat(__fsub_rn(g1, q1.x), q1.y);
    v0 = dot_halves(~rnd, 0x0001u, __float_as_uint(__fmaf_rn(p0, 65536.0f, kMagic)) + (k0 << 13));
    v1 = dot_halves(~rnd, 0x0100u, __float_as_uint(__fmaf_rn(p1, 65536.0f, kMagic)) + (k1 << 13));
}
__device__ __forceinline__ void code_grid2(float g0, float g1, f32x2 alpha2, float inv_2alpha, f32x2 cell_scale2, const char* s_grid,
                                           const char* s_cell, uint32_t rnd, uint32_t& v0, uint32_t& v1) {
    const f32x2 g = pair(g0, g1);
    float s0, s1;
    unpair(add2(g, alpha2), s0, s1);
    // cell = floor(M * sat((g + alpha) * inv_2alpha)) as a denormal whose bit pattern is the integer; * 8 = byte offset
    const f32x2 cell8 = mul2(mul2_rd(pair(mul_sat(s0, inv_2alpha), mul_sat(s1, inv_2alpha)), cell_scale2), both(8.0f));
    float c0, c1;
    unpair(cell8, c0, c1);
    const float2 gc0 = *reinterpret_cast<const float2*>(s_grid + __float_as_uint(c0));
    const float2 gc1 = *reinterpret_cast<const float2*>(s_grid + __float_as_uint(c1));
    code_cells2(g0, g1, gc0, gc1, s_cell, rnd, v0, v1);
}

// The same through a logarithmic grid, whose cells are the exponent and the four highest mantissa bits of |g|, 16 per binade,
// mirrored for negative values.  Levels 1/16 apart, relatively, are in different cells, however small they are against alpha:
// this serves the codebooks of heavy tails (exponent 2.5, 16 levels, alpha at 10^4 g_min), whose inner levels are closer
// than 1/2048 of the range.  Its index arithmetic takes 4.5 operations of the integer / compare pipe per element where the
// linear grid's floor takes as many of the multiply-add pipes, which have more room, so the linear grid goes first.
// 25.6 M x 16, 16 levels, exponent 2.5: 575 us by binary search, 366 this way (device parameters 579, 404); where both grids
// serve, exponent 3: 327 us linear, 379 logarithmic; 250 M x 4, 8 levels 782 and 874.
// The high half of a float, without its three lowest bits, is 8 times its cell: the byte offset of an 8-byte entry.  Two values
// at a time in the halves of a word.  t = max(g, -alpha): a NaN takes the lowest cell and code 0.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {          // with sign replication, unlike __byte_perm
    uint32_t r; asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel)); return r;
}
__host__ __device__ inline uint32_t log_cell8(uint32_t bits) { return (bits >> 16) & 0x7FF8u; }
__device__ __forceinline__ void code_log2(float g0, float g1, float alpha, uint32_t nbase2, uint32_t top2, const char* s_middle,
                                          const char* s_cell, uint32_t rnd, uint32_t& v0, uint32_t& v1) {
    const float t0 = fmaxf(g0, -alpha), t1 = fmaxf(g1, -alpha);
    const uint32_t y = __byte_perm(__float_as_uint(t0), __float_as_uint(t1), 0x7632u);
    const uint32_t z = __viaddmin_s16x2_relu(y & 0x7FF87FF8u, nbase2, top2) ^ (prmt(y, y, 0xBB99u) & 0xFFF8FFF8u);
    const float2 gc0 = *reinterpret_cast<const float2*>(s_middle + static_cast<int>(prmt(z, z, 0x9910u)));
    const float2 gc1 = *reinterpret_cast<const float2*>(s_middle + static_cast<int>(prmt(z, z, 0xBB32u)));
    code_cells2(t0, t1, gc0, gc1, s_cell, rnd, v0, v1);
}

// General codebook by branch-free binary search (used when no grid of at most kMaxGridCells cells
// separates the levels): search[] holds l_1 .. l_{s-1} at indices 1 .. s-1 and +inf from index s on.
template <int BITS>
__device__ __forceinline__ float code_binary(float g, float alpha, const float* search, const float2* cell, float rf) {
    const float t = fminf(fmaxf(g, -alpha), alpha);   // NaN -> -alpha
    uint32_t k = 0;
#pragma unroll
    for (int step = (1 << BITS) >> 1; step > 0; step >>= 1)
        if (t >= search[k + step]) k += step;
    const float2 c = cell[k];
    const float p = __fmul_rn(__fsub_rn(t, c.x), c.y);
    return __fadd_rn(static_cast<float>(k), rounds_up(p, rf));
}

// Four pairs of float codes (elements 0..7 of a group, each code < 2^BITS) -> their 8*BITS packed
// bits, LSB first.  Every partial sum is an integer below 2^24, so the fp32 arithmetic is exact.
// Returns a word whose low 8*BITS bits are the packed codes.
template <int BITS>
__device__ __forceinline__ uint32_t pack8(const f32x2 (&c)[4]) {
    constexpr float B = static_cast<float>(1 << BITS), B2 = B * B;
    if constexpr (BITS <= 3) {
        f32x2 a = fma2(c[3], both(B2), c[2]);
        a = fma2(a, both(B2), c[1]);
        a = fma2(a, both(B2), c[0]);
        float ev, od;
        unpair(a, ev, od);
        return __float2uint_rz(__fmaf_rn(od, B, ev));
    } else {
        float e0, o0, e1, o1;
        unpair(fma2(c[1], both(B2), c[0]), e0, o0);       // elements 0..3: 16 bits
        unpair(fma2(c[3], both(B2), c[2]), e1, o1);       // elements 4..7: 16 bits
        return __float2uint_rz(__fmaf_rn(o0, B, e0)) + (__float2uint_rz(__fmaf_rn(o1, B, e1)) << 16);
    }
}

// The cell of a level, counted from the middle (negative below it), and whether the grid's cells separate the levels: each cell
// holds at most one, and there are at most kMaxGridCells.  A level 0 is left to the search: -0 is below its cell.
__host__ __device__ inline uint32_t float_bits(float x) {
#ifdef __CUDA_ARCH__
    return __float_as_uint(x);
#else
    uint32_t b;
    memcpy(&b, &x, 4);
    return b;
#endif
}
__host__ __device__ inline uint32_t log_cell(float level, uint32_t base8) {
    const uint32_t b = float_bits(level), z = (log_cell8(b) - base8) >> 3;
    return b >> 31 ? ~z : z;
}

struct RunCtx {
    float alpha, inv_step, top, inv_2alpha, cell_scale;
    uint32_t log_nbase2, log_top2;             // logarithmic grid; s_grid is then its middle
    UniformQ u;
    const char* s_grid; const char* s_cell; const float* s_search;
};

template <int BITS>
__device__ __forceinline__ UniformQ uniform_q(const WorkerQ& q) {
    constexpr float L = static_cast<float>(1 << BITS);
    return UniformQ{q.inv_step_l, (L - 1.0f) / L, both(L * 65536.0f)};
}

template <int BITS, int SEARCH>
__device__ __forceinline__ RunCtx run_ctx(const WorkerQ& q, const float2* s_grid, const float2* s_cell, const float* s_search) {
    const uint32_t n = SEARCH == kLogGrid ? q.log_cells : 0u;
    return RunCtx{q.alpha, q.inv_step, q.top, q.inv_2alpha, q.cell_scale, ((0u - q.log_base) & 0xFFFFu) * 0x00010001u, 8u * (n - 1) * 0x00010001u,
                  uniform_q<BITS>(q), reinterpret_cast<const char*>(s_grid + n), reinterpret_cast<const char*>(s_cell), s_search};
}

// inv_step / L for the scaled uniform path: exact when the quotient is a normal number (L is a power of
// two); 0 tells the launch to use the unscaled arithmetic instead.  Same expression on host and device.
__host__ __device__ inline float scaled_inv_step(float inv_step, uint32_t num_levels) {
    const float q = inv_step / static_cast<float>(num_levels);
    return (q >= 1.17549435e-38f && q <= 3.402823466e38f) ? q : 0.0f;
}

// the 16 random bits of slot e of a Philox block, as the float 2^23 + r
__device__ __forceinline__ float slot_as_float(const uint32_t (&rnd)[4], int e) {
    return __uint_as_float(__byte_perm(rnd[e >> 1], kMagicBits, (e & 1) ? 0x7432u : 0x7410u));
}

// The arithmetic of one run of 32 elements that are already in registers: quantize, pack, store.
template <int BITS, int SEARCH, bool BF16>
__device__ __forceinline__ void quantize_run(const Raw8<BF16> (&g)[4], uint32_t* prow, uint64_t run, uint32_t worker,
                                             const RoundKeys& rk, const RunCtx& cx) {
    const uint64_t j0 = run << 5;
    const uint32_t blk_lo = static_cast<uint32_t>(j0 >> 3);
    const PhiloxRun pr = philox_run(static_cast<uint32_t>(j0 >> 35), worker, rk);
    const f32x2 alpha2 = both(cx.alpha), inv_step2 = both(cx.inv_step), cell_scale2 = both(cx.cell_scale);
    uint32_t chunk[4];   // the 8*BITS packed bits of each group
#pragma unroll
    for (int grp = 0; grp < 4; ++grp) {
        uint32_t rnd[4];
        philox_block(blk_lo + grp, pr, rk, rnd);                      // j0 >> 3 is a multiple of 4: no carry
        if constexpr (SEARCH == kUniform || SEARCH == kGrid || SEARCH == kLogGrid) {
            uint32_t v[8];                       // the codes in byte 2
#pragma unroll
            for (int h = 0; h < 4; ++h) {        // elements 2h, 2h+1 of the group
                if constexpr (SEARCH == kUniform) {
                    float sum0, sum1;
                    pair_plus_alpha<BF16>(g[grp], h, cx.alpha, sum0, sum1);
                    code_uniform2<BF16>(sum0, sum1, cx.u, rnd[h], v[2 * h], v[2 * h + 1]);
                } else {
                    const float g0 = elem<BF16>(g[grp], 2 * h), g1 = elem<BF16>(g[grp], 2 * h + 1);
                    if constexpr (SEARCH == kGrid)
                        code_grid2(g0, g1, alpha2, cx.inv_2alpha, cell_scale2, cx.s_grid, cx.s_cell, rnd[h], v[2 * h], v[2 * h + 1]);
                    else code_log2(g0, g1, cx.alpha, cx.log_nbase2, cx.log_top2, cx.s_grid, cx.s_cell, rnd[h], v[2 * h], v[2 * h + 1]);
                }
            }
            chunk[grp] = pack_byte2<BITS>(v);
        } else {
            f32x2 code[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int e = 2 * h;
                const float rf0 = slot_as_float(rnd, e), rf1 = slot_as_float(rnd, e + 1);
                if constexpr (SEARCH == kUniformWide) {
                    float sum0, sum1;
                    pair_plus_alpha<BF16>(g[grp], h, cx.alpha, sum0, sum1);
                    code[h] = code_uniform2_wide(sum0, sum1, inv_step2, cx.top, rf0, rf1);
                } else {
                    const float g0 = elem<BF16>(g[grp], e), g1 = elem<BF16>(g[grp], e + 1);
                    code[h] = pair(code_binary<BITS>(g0, cx.alpha, cx.s_search, reinterpret_cast<const float2*>(cx.s_cell), rf0),
                                   code_binary<BITS>(g1, cx.alpha, cx.s_search, reinterpret_cast<const float2*>(cx.s_cell), rf1));
                }
            }
            chunk[grp] = pack8<BITS>(code);
        }
    }

    // four chunks of 8*BITS bits -> BITS words, LSB first
    uint32_t w[BITS];
    if constexpr (BITS == 4) { w[0] = chunk[0]; w[1] = chunk[1]; w[2] = chunk[2]; w[3] = chunk[3]; }
    if constexpr (BITS == 3) {
        w[0] = chunk[0] | (chunk[1] << 24);
        w[1] = (chunk[1] >> 8) | (chunk[2] << 16);
        w[2] = (chunk[2] >> 16) | (chunk[3] << 8);
    }
    if constexpr (BITS == 2) { w[0] = __byte_perm(chunk[0], chunk[1], 0x5410u); w[1] = __byte_perm(chunk[2], chunk[3], 0x5410u); }
    if constexpr (BITS == 1) { w[0] = chunk[0] | (chunk[1] << 8) | (chunk[2] << 16) | (chunk[3] << 24); }

    uint32_t* dst = prow + run * BITS;
    if constexpr (BITS == 4) *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
    if constexpr (BITS == 3) { dst[0] = w[0]; dst[1] = w[1]; dst[2] = w[2]; }
    if constexpr (BITS == 2) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
    if constexpr (BITS == 1) dst[0] = w[0];
}

// One whole run: load, quantize, pack, store.
template <int BITS, int SEARCH, bool BF16>
__device__ __forceinline__ void compress_run(const char* row, uint32_t* prow, uint64_t run, uint32_t worker, const RoundKeys& rk,
                                             const RunCtx& cx) {
    constexpr size_t esz = BF16 ? 2 : 4;
    Raw8<BF16> g[4];
#pragma unroll
    for (int grp = 0; grp < 4; ++grp) load8_raw<BF16>(row + ((run << 5) + 8 * grp) * esz, g[grp]);
    quantize_run<BITS, SEARCH, BF16>(g, prow, run, worker, rk, cx);
}

// A row's last run, possibly partial, by one warp: a lane takes one element, with the decision in its plain form (clip,
// interval, p, T, code = k + [r < T]); bits beyond the row's end and the padding words are zero.
template <int BITS, bool UNIFORM, bool BF16>
__device__ __forceinline__ void compress_last_run(const char* row, uint32_t* prow, uint64_t d, uint32_t worker, const RoundKeys& rk,
                                                  const WorkerQ& q) {
    constexpr int s = (1 << BITS) - 1;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t run = (d - 1) >> 5, j = (run << 5) + lane;
    uint32_t code = 0;
    if (j < d) {
        const float t = fminf(fmaxf(load1<BF16>(row, j), -q.alpha), q.alpha);      // NaN -> -alpha
        float k = 0.0f, p;
        if constexpr (UNIFORM) {
            const float x = __fmul_rn(__fadd_rn(t, q.alpha), q.inv_step);
            k = fminf(floorf(x), static_cast<float>(s - 1));
            p = __fsub_rn(x, k);
        } else {
            int i = 0;
            for (int l = 1; l < s; ++l)
                if (q.levels[l] <= t) i = l;
            k = static_cast<float>(i);
            p = __fmul_rn(__fsub_rn(t, q.levels[i]), q.inv_width[i]);
        }
        uint32_t rnd[4];
        philox_block(static_cast<uint32_t>(j >> 3), philox_run(static_cast<uint32_t>(j >> 35), worker, rk), rk, rnd);
        const uint32_t word = (lane & 4u) ? ((lane & 2u) ? rnd[3] : rnd[2]) : ((lane & 2u) ? rnd[1] : rnd[0]);
        const uint32_t r = (lane & 1u) ? word >> 16 : word & 0xFFFFu;
        code = static_cast<uint32_t>(k + rounds_up(p, __uint_as_float(kMagicBits | r)));
    }
    const uint64_t at = static_cast<uint64_t>(code) << ((lane * BITS) & 31u);
    const uint32_t w = (lane * BITS) >> 5;
    const uint64_t first = run * BITS, words_out = (((d * BITS + 31) >> 5) + 3) & ~static_cast<uint64_t>(3);
#pragma unroll
    for (uint32_t i = 0; i < BITS; ++i) {
        const uint32_t bits = __reduce_or_sync(0xFFFFFFFFu, (w == i ? static_cast<uint32_t>(at) : 0u) | (w + 1 == i ? static_cast<uint32_t>(at >> 32) : 0u));
        if (lane == i && first + i < words_out) prow[first + i] = bits;
    }
    if (first + BITS + lane < words_out) prow[first + BITS + lane] = 0u;             // at most three words of padding
}

#ifndef TQ_COMPRESS_MIN_BLOCKS
#define TQ_COMPRESS_MIN_BLOCKS 4
#endif

// Per-block set-up of the shared tables for quantizer q (ends with a block barrier unless the codebook is uniform).
// s_grid must hold kMaxGridCells + 1 entries when SEARCH is a grid.  LANES: a lane per level, for fp32 rows with 16 levels in device memory, where fourteen
// comparisons per cell show in the start of a row (3.5 M x 1 7.25 -> 7.11 us, 2 M x 4 11.56 -> 11.38, 250 M x 4 984 -> 979).  Elsewhere it is the slower form: bf16
// rows and fewer levels (64 x 547 k bf16 in 16 groups, 16 / 8 / 4 levels 49.2 / 46.2 / 45.7 us, with it 51.1 / 48.1 / 46.3; 1 M x 1 fp32, 8 levels 3.9, with it
// 4.3), and the host's parameters, whose tables are built while the kernel before still runs and whose main loop gets other registers (25.6 M x 16, 16
// levels: 310 -> 322 us).
template <int BITS, int SEARCH, bool LANES>
__device__ __forceinline__ void build_tables(const WorkerQ& q, float2* s_grid, float2* s_cell, float* s_search) {
    constexpr int L = 1 << BITS;
    if constexpr (!is_uniform(SEARCH)) {
        if (threadIdx.x < L - 1) s_cell[threadIdx.x] = make_float2(q.levels[threadIdx.x], q.inv_width[threadIdx.x]);
    }
    if constexpr (SEARCH == kBinary) {
        if (threadIdx.x < 2 * TQ_MAX_LEVELS)
            s_search[threadIdx.x] = (threadIdx.x >= 1 && threadIdx.x <= L - 2) ? q.levels[threadIdx.x] : __int_as_float(0x7F800000);
    }
    constexpr bool kCells = SEARCH == kGrid || SEARCH == kLogGrid;
    if constexpr (kCells && LANES) {
        // A lane for each interior level l_1 .. l_{s-1} (their cells are distinct and in order, or the grid would not have been chosen); a warp fills
        // in 32 cells at a time, most of which hold none.
        const uint32_t lane = threadIdx.x & 31u;
        const bool interior = lane >= 1 && lane <= L - 2;
        const float level = lane < L ? q.levels[lane] : 0.0f;
        const uint32_t cell = SEARCH == kGrid ? __float_as_uint(grid_cell(level, q.alpha, q.inv_2alpha, q.cell_scale)) : log_cell(level, q.log_base) + q.log_cells;
        const uint32_t last = SEARCH == kGrid ? q.cells : 2 * q.log_cells - 1;
        for (uint32_t c0 = threadIdx.x - lane; c0 <= last; c0 += kThreads) {
            const uint32_t c = c0 + lane;
            uint32_t below = __popc(__ballot_sync(0xFFFFFFFFu, interior && cell < c0));
            float boundary = __int_as_float(0x7FC00000);               // NaN: no value compares >= it
            for (uint32_t here = __ballot_sync(0xFFFFFFFFu, interior && cell - c0 < 32u); here != 0; here &= here - 1) {
                const int j = __ffs(static_cast<int>(here)) - 1;
                const uint32_t at = __shfl_sync(0xFFFFFFFFu, cell, j);
                const float l = __shfl_sync(0xFFFFFFFFu, level, j);
                if (at < c) ++below;
                if (at == c) boundary = l;
            }
            if (c <= last) s_grid[c] = make_float2(boundary, __uint_as_float(8 * below));
        }
    } else if constexpr (kCells) {
        // cells of the interior levels l_1 .. l_{s-1} (distinct, or the grid would not have been chosen)
        uint32_t lc[L];
#pragma unroll
        for (int j = 1; j <= L - 2; ++j)
            lc[j] = SEARCH == kGrid ? __float_as_uint(grid_cell(q.levels[j], q.alpha, q.inv_2alpha, q.cell_scale))
                                    : log_cell(q.levels[j], q.log_base) + q.log_cells;
        const uint32_t last = SEARCH == kGrid ? q.cells : 2 * q.log_cells - 1;
        for (uint32_t c = threadIdx.x; c <= last; c += kThreads) {
            uint32_t below = 0;                                        // 8 times their number
            float boundary = __int_as_float(0x7FC00000);               // NaN: no value compares >= it
#pragma unroll
            for (int j = 1; j <= L - 2; ++j) {
                if (lc[j] < c) below += 8u;
                if (lc[j] == c) boundary = q.levels[j];
            }
            s_grid[c] = make_float2(boundary, __uint_as_float(below));
        }
    }
    if constexpr (!is_uniform(SEARCH)) __syncthreads();
}

// Quantizers passed by value in the kernel's parameter space (host-side tq_params).
template <int BITS, int SEARCH, bool BF16, uint32_t N>
__global__ void __launch_bounds__(kThreads, TQ_COMPRESS_MIN_BLOCKS)
compress_kernel(const void* __restrict__ grad, uint64_t d, uint64_t grad_stride,
                const __grid_constant__ CompressArgs<N> args, const __grid_constant__ RoundKeys rk,
                uint32_t first_worker, uint32_t* __restrict__ packed, uint64_t words_stride) {
    __shared__ __align__(16) float2 s_grid[SEARCH == kGrid || SEARCH == kLogGrid ? kMaxGridCells + 1 : 1];
    __shared__ __align__(16) float2 s_cell[TQ_MAX_LEVELS];
    __shared__ float s_search[2 * TQ_MAX_LEVELS];
    constexpr size_t esz = BF16 ? 2 : 4;
    const WorkerQ& q = args.q[blockIdx.y];
    const uint32_t worker = first_worker + blockIdx.y;
    const char* row = static_cast<const char*>(grad) + static_cast<uint64_t>(blockIdx.y) * grad_stride * esz;
    uint32_t* prow = packed + static_cast<uint64_t>(blockIdx.y) * words_stride;
    build_tables<BITS, SEARCH, false>(q, s_grid, s_cell, s_search);          // from kernel parameters: before the wait
    pdl_wait();
    const RunCtx cx = run_ctx<BITS, SEARCH>(q, s_grid, s_cell, s_search);
    const uint64_t whole = (d - 1) >> 5, stride = static_cast<uint64_t>(gridDim.x) * kThreads;     // runs before the row's last one are whole
    for (uint64_t run = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x; run < whole; run += stride)
        compress_run<BITS, SEARCH, BF16>(row, prow, run, worker, rk, cx);
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x < 32) compress_last_run<BITS, is_uniform(SEARCH), BF16>(row, prow, d, worker, rk, q);
}

// The grid cell of a value as a plain integer (device copy of the host's cell_of).
__device__ __forceinline__ uint32_t cell_index(float g, float alpha, float inv_2alpha, uint32_t cells) {
    return __float_as_uint(grid_cell(g, alpha, inv_2alpha, __uint_as_float(cells)));   // M * 2^-149 has bit pattern M
}

// Quantizers read from device memory (tq_params_device): no host round trip before the launch.
// The block turns a job's tq_params_t into the kernel's WorkerQ, including the choice of the lookup grid.  Ends with a
// block barrier.
template <int BITS, bool NONUNIFORM>
__device__ __forceinline__ void load_worker(const tq_params_t& p, WorkerQ& s_q) {
    if (threadIdx.x < 32) {
        const uint32_t lane = threadIdx.x;
        if (lane < TQ_MAX_LEVELS) {
            s_q.levels[lane] = p.levels[lane];
            s_q.inv_width[lane] = p.inv_width[lane];
        }
        const float alpha = p.alpha, inv_step = p.inv_step;
        const bool ok = alpha > 0.0f && p.bits == BITS && !(p.flags & TQ_FLAG_INVALID);
        __syncwarp();
        const float inv_2alpha = ok ? __fdiv_rn(1.0f, __fmul_rn(2.0f, alpha)) : 0.0f;
        uint32_t cells = 0, log_base = 0, log_cells = 0;
        if constexpr (NONUNIFORM) {      // choose_cells, a lane for each interior level
            constexpr int s = (1 << BITS) - 1;
            const bool mine = lane >= 2 && lane <= s - 1;
            const uint32_t cell = lane < TQ_MAX_LEVELS ? cell_index(s_q.levels[lane], alpha, inv_2alpha, kMaxGridCells) : 0u;
            const uint32_t prev = __shfl_up_sync(0xFFFFFFFFu, cell, 1);
            const uint32_t drop = __reduce_min_sync(0xFFFFFFFFu, mine && cell > prev ? 31u - __clz(static_cast<int>(cell ^ prev)) : 31u);
            const bool distinct = !__any_sync(0xFFFFFFFFu, mine && cell <= prev) && ok && inv_2alpha <= 3.402823466e38f;
            const uint32_t m = drop >= 31 ? 0u : static_cast<uint32_t>(kMaxGridCells) >> drop;
            if (distinct) cells = m < static_cast<uint32_t>(kMinGridCells) ? kMinGridCells : m;
            else if (ok) {               // choose_log_grid
                const bool interior = lane >= 1 && lane <= s - 1;
                const float level = lane < TQ_MAX_LEVELS ? s_q.levels[lane] : 0.0f;
                const uint32_t c8 = log_cell8(__float_as_uint(level));
                log_base = __reduce_min_sync(0xFFFFFFFFu, interior ? c8 : 0x7FF8u);
                const uint32_t n = ((__reduce_max_sync(0xFFFFFFFFu, interior ? c8 : 0u) - log_base) >> 3) + 1;
                const int lc = static_cast<int>(log_cell(level, log_base)), below = __shfl_up_sync(0xFFFFFFFFu, lc, 1);
                const bool bad = (interior && level == 0.0f) || (mine && lc <= below) || n > kMaxGridCells / 2;
                if (!__any_sync(0xFFFFFFFFu, bad)) log_cells = n;
            }
        }
        if (lane == 0) {
            s_q.alpha = ok ? alpha : 0.0f;
            s_q.inv_step = inv_step;
            s_q.inv_step_l = scaled_inv_step(inv_step, 1u << BITS);
            s_q.top = static_cast<float>((1 << BITS) - 1);
            s_q.inv_2alpha = inv_2alpha;
            s_q.cells = cells; s_q.log_base = log_base; s_q.log_cells = log_cells;
            s_q.cell_scale = __uint_as_float(cells);
        }
    }
    __syncthreads();
}

// What a block of the device-parameter kernel keeps in shared memory.  Its place in its range of pieces is there too, and
// is read back where it is needed, so that the loop over a piece's runs has the registers to itself.
template <bool NONUNIFORM>
struct BlockState {
    float2 grid[NONUNIFORM ? kMaxGridCells + 1 : 1];
    float2 cell[TQ_MAX_LEVELS];
    float search[2 * TQ_MAX_LEVELS];
    WorkerQ q;
    JobPiece piece;
    uint64_t cur, end;
};

// The piece in sh.piece.
template <int BITS, int SEARCH, bool BF16, class State>
__device__ __forceinline__ void compress_piece(State& sh, const void* __restrict__ grad, uint64_t grad_stride, const RoundKeys& rk,
                                               uint32_t first_worker, uint32_t* __restrict__ packed, uint64_t words_stride,
                                               const TilePlan& plan) {
    constexpr size_t esz = BF16 ? 2 : 4;
    build_tables<BITS, SEARCH, !BF16 && BITS == 4>(sh.q, sh.grid, sh.cell, sh.search);
    const RunCtx cx = run_ctx<BITS, SEARCH>(sh.q, sh.grid, sh.cell, sh.search);
    const char* row = static_cast<const char*>(grad) + (static_cast<uint64_t>(sh.piece.worker) * grad_stride + sh.piece.off) * esz;
    uint32_t* prow = packed + static_cast<uint64_t>(sh.piece.worker) * words_stride + plan.segs.woff[sh.piece.seg];
    const uint32_t worker = first_worker + sh.piece.worker;
    const uint64_t whole = (sh.piece.d - 1) >> 5, stop = sh.piece.tile1 * kThreads;       // runs before the row's last one are whole
    const uint64_t end = stop < whole ? stop : whole;
    // from the piece's end to its beginning: what the statistics pass before this one read last is still in L2
    const uint64_t begin = sh.piece.tile0 * kThreads + threadIdx.x;
    if (begin < end)
        for (uint64_t run = begin + (end - 1 - begin) / kThreads * kThreads;; run -= kThreads) {
            compress_run<BITS, SEARCH, BF16>(row, prow, run, worker, rk, cx);
            if (run == begin) break;
        }
    if (sh.piece.last && threadIdx.x < 32) compress_last_run<BITS, is_uniform(SEARCH), BF16>(row, prow, sh.piece.d, worker, rk, sh.q);
}

// The same for a quantizer that needs one of the rare arithmetics (levels that no grid separates: binary search; alpha too
// large for the scaled inverse step).  Out of line, so that it costs the common loop no registers: as a second kernel
// behind the first, which nearly always found nothing to do, it was 2-3 us of every call.
template <int BITS, int SEARCH, bool BF16, class State>
__device__ __noinline__ void compress_piece_rare(State& sh, const void* grad, uint64_t grad_stride, const RoundKeys& rk, uint32_t first_worker,
                                                 uint32_t* packed, uint64_t words_stride, const TilePlan& plan) {
    compress_piece<BITS, SEARCH, BF16>(sh, grad, grad_stride, rk, first_worker, packed, words_stride, plan);
}

// The block's pieces of the jobs -- workers, or (worker, segment) pairs, see TilePlan; a tile is one run per thread.
// Rows of jobs that are marked invalid (alpha = 0) become all code 0.
// BEHIND: behind the decision-table kernel, for the rows that it does not serve.
template <int BITS, bool NONUNIFORM, bool BF16, bool BEHIND>
__global__ void __launch_bounds__(kThreads, TQ_COMPRESS_MIN_BLOCKS)
compress_kernel_dev(const void* __restrict__ grad, uint64_t grad_stride, const tq_params_t* params,
                    const __grid_constant__ RoundKeys rk, uint32_t first_worker, uint32_t* __restrict__ packed, uint64_t words_stride,
                    const __grid_constant__ TilePlan plan, uint32_t n_jobs) {
    __shared__ __align__(16) BlockState<NONUNIFORM> sh;
    if (threadIdx.x == 0) {                                    // the first piece, before the wait; no block is empty
        uint64_t cur = first_tile_of_block(plan, blockIdx.x);
        sh.end = first_tile_of_block(plan, blockIdx.x + 1);
        sh.piece = next_piece(plan, cur, sh.end);
        sh.cur = cur;
    }
    pdl_wait();
    if constexpr (BEHIND) {              // nearly always nothing is left, which one look over all records shows
        bool left = false;
        for (uint32_t j = threadIdx.x; j < n_jobs; j += kThreads) left = left || !lut_serves_record(params[j], BITS);
        if (!__syncthreads_or(left)) return;
    }
    while (true) {
        __syncthreads();                 // the piece is known
        const tq_params_t& p = params[sh.piece.job];
        if (!BEHIND || !lut_serves_record(p, BITS)) {        // same rule, evaluated by every thread
            load_worker<BITS, NONUNIFORM>(p, sh.q);
            if (!(sh.q.alpha > 0.0f)) {
                uint32_t* prow = packed + static_cast<uint64_t>(sh.piece.worker) * words_stride + plan.segs.woff[sh.piece.seg];
                const uint64_t words_out = (((sh.piece.d * BITS + 31) >> 5) + 3) & ~static_cast<uint64_t>(3);
                const uint64_t w1 = sh.piece.last ? words_out : sh.piece.tile1 * kThreads * BITS;
                for (uint64_t w = sh.piece.tile0 * kThreads * BITS + threadIdx.x; w < w1; w += kThreads) prow[w] = 0u;
            } else if (NONUNIFORM && sh.q.cells == 0 && sh.q.log_cells != 0) {
                compress_piece_rare<BITS, kLogGrid, BF16>(sh, grad, grad_stride, rk, first_worker, packed, words_stride, plan);
            } else if (NONUNIFORM && sh.q.cells == 0) {
                compress_piece_rare<BITS, kBinary, BF16>(sh, grad, grad_stride, rk, first_worker, packed, words_stride, plan);
            } else if (!NONUNIFORM && sh.q.inv_step_l == 0.0f) {
                compress_piece_rare<BITS, kUniformWide, BF16>(sh, grad, grad_stride, rk, first_worker, packed, words_stride, plan);
            } else {
                compress_piece<BITS, NONUNIFORM ? kGrid : kUniform, BF16>(sh, grad, grad_stride, rk, first_worker, packed, words_stride, plan);
            }
        }
        if (sh.cur >= sh.end) return;
        __syncthreads();                 // the piece has been served
        if (threadIdx.x == 0) {
            uint64_t cur = sh.cur;
            sh.piece = next_piece(plan, cur, sh.end);
            sh.cur = cur;
        }
    }
}

// ---- host side ---------------------------------------------------------------------------------------

// Smallest power-of-two grid (32 .. 2048 cells) that puts the interior levels in distinct cells; 0 if none.  The cell of a
// level is exactly what grid_cell() computes on the device: every step is a single IEEE operation (u * M is exact for M a
// power of two), and the cell in a grid 2^k times coarser is the cell in the finest one without its last k bits.
static uint32_t choose_cells(const tq_params_t& p, float inv_2alpha) {
    const int s = static_cast<int>(p.num_levels) - 1;
    uint32_t prev = 0;
    int drop = 31;                       // bits that may go: up to the highest one in which neighbours differ
    for (int j = 1; j <= s - 1; ++j) {
        float u = (p.levels[j] + p.alpha) * inv_2alpha;
        u = !(u > 0.0f) ? 0.0f : (u > 1.0f ? 1.0f : u);
        const uint32_t cell = static_cast<uint32_t>(u * static_cast<float>(kMaxGridCells));
        if (j > 1) {
            if (cell <= prev) return 0;
            const int top = 31 - __builtin_clz(cell ^ prev);
            drop = top < drop ? top : drop;
        }
        prev = cell;
    }
    const uint32_t m = drop >= 31 ? 0u : static_cast<uint32_t>(kMaxGridCells) >> drop;
    return m < static_cast<uint32_t>(kMinGridCells) ? kMinGridCells : m;
}

// The logarithmic grid of a codebook: 8 * its first cell, and its cells per sign, 0 if it does not separate the levels.
static uint32_t choose_log_grid(const tq_params_t& p, uint32_t* base8) {
    const int s = static_cast<int>(p.num_levels) - 1;
    uint32_t lo = 0x7FF8u, hi = 0;
    for (int j = 1; j <= s - 1; ++j) {
        const uint32_t c8 = log_cell8(float_bits(p.levels[j]));
        lo = c8 < lo ? c8 : lo;
        hi = c8 > hi ? c8 : hi;
        if (p.levels[j] == 0.0f) return 0;
    }
    *base8 = lo;
    for (int j = 2; j <= s - 1; ++j)
        if (static_cast<int>(log_cell(p.levels[j], lo)) <= static_cast<int>(log_cell(p.levels[j - 1], lo))) return 0;
    const uint32_t n = s > 1 ? ((hi - lo) >> 3) + 1 : 0;
    return n > kMaxGridCells / 2 ? 0 : n;
}

// Shares per resident block when each would get `tiles` tiles as one share: the hardware hands the later ones to the blocks
// that finish first, which evens out SMs and the blocks of an SM, as long as a share repays its set-up.  Device parameters, 1 / 2 /
// 4 / 8 shares: 25.6 M x 16 (84 tiles) 339 / 327 / 324 / 328 us, 11.2 M x 8 (18 tiles) 70 / 69 / 65 / 68, 1 M x 64 (13) 50 / 48 / 51 / 55,
// 4 M x 4 (3) 19.8 / 19.7 / 21.4 / 21.4, 124 M x 8 bf16 uniform 541 / 519 / 511 / 513.
static uint64_t ranges_per_block(uint64_t tiles) {
    const uint64_t n = tiles / 5;
    return n < 1 ? 1 : n > 6 ? 6 : n;
}

// Persistent grid: 4 resident blocks per SM spread over the workers (table modes build their lookup
// grid once per block); uniform mode has no per-block set-up, so one block per tile lets the hardware
// scheduler balance the tail.
static dim3 compress_grid(uint64_t d, uint32_t n_workers, bool persistent) {
    const uint64_t n_runs = (d + 31) >> 5;
    const uint64_t tiles = (n_runs + kThreads - 1) / kThreads;
    uint64_t per_worker = static_cast<uint64_t>(sm_count()) * TQ_COMPRESS_MIN_BLOCKS / n_workers;   // rounded down: one wave holds the grid
    if (persistent && per_worker > 0) per_worker *= ranges_per_block(tiles / per_worker);
    if (!persistent || per_worker > tiles) per_worker = tiles;
    if (per_worker > 0x7FFFFFFFull) per_worker = 0x7FFFFFFFull;
    if (per_worker < 1) per_worker = 1;
    return dim3(static_cast<unsigned>(per_worker), n_workers);
}

template <int BITS, int SEARCH, bool BF, uint32_t N>
static cudaError_t launch(const CompressCall& c, const CompressArgs<N>& args, dim3 grid) {
    return launch_kernel(compress_kernel<BITS, SEARCH, BF, N>, grid, kThreads, 0, c.stream, c.grad, c.d, c.grad_stride, args, round_keys(c.seed),
                         c.first_worker, c.packed, c.words_stride);
}

template <int BITS>
static cudaError_t dispatch(const CompressCall& c, const CompressArgs<TQ_MAX_WORKERS>& a, dim3 grid, int search) {
    const bool few = c.n_workers <= kFewWorkers;
    const CompressArgs<kFewWorkers>& f = reinterpret_cast<const CompressArgs<kFewWorkers>&>(a);      // its first entries
    if (search == kGrid) {
        if (few) return c.bf16 ? launch<BITS, kGrid, true>(c, f, grid) : launch<BITS, kGrid, false>(c, f, grid);
        return c.bf16 ? launch<BITS, kGrid, true>(c, a, grid) : launch<BITS, kGrid, false>(c, a, grid);
    }
    if (search == kLogGrid) return c.bf16 ? launch<BITS, kLogGrid, true>(c, a, grid) : launch<BITS, kLogGrid, false>(c, a, grid);
    if (search == kBinary) return c.bf16 ? launch<BITS, kBinary, true>(c, a, grid) : launch<BITS, kBinary, false>(c, a, grid);
    if (search == kUniformWide) return c.bf16 ? launch<BITS, kUniformWide, true>(c, a, grid) : launch<BITS, kUniformWide, false>(c, a, grid);
    if (few) return c.bf16 ? launch<BITS, kUniform, true>(c, f, grid) : launch<BITS, kUniform, false>(c, f, grid);
    return c.bf16 ? launch<BITS, kUniform, true>(c, a, grid) : launch<BITS, kUniform, false>(c, a, grid);
}

cudaError_t launch_compress(const CompressCall& c) {
    if (c.d == 0 && !c.segs) return cudaSuccess;
    if (c.params_dev) return launch_compress_dev(c);
    {
        bool applied = false;
        const cudaError_t e = launch_compress_lut(c, &applied);
        if (applied || e != cudaSuccess) return e;
    }
    static thread_local CompressArgs<TQ_MAX_WORKERS> args;   // 9 KB: keep it off the stack
    int search = c.nonuniform ? kGrid : kUniform;
    for (uint32_t i = 0; i < c.n_workers; ++i) {
        const tq_params_t& p = c.params[i];
        WorkerQ& q = args.q[i];
        q.alpha = p.alpha; q.inv_step = p.inv_step; q.top = static_cast<float>(p.num_levels - 1);
        q.inv_2alpha = 1.0f / (2.0f * p.alpha);
        q.inv_step_l = scaled_inv_step(p.inv_step, p.num_levels);
        if (!c.nonuniform && q.inv_step_l == 0.0f) search = kUniformWide;
        q.cells = q.log_base = q.log_cells = 0; q.cell_scale = 0.0f;
        for (int k = 0; k < TQ_MAX_LEVELS; ++k) { q.levels[k] = p.levels[k]; q.inv_width[k] = p.inv_width[k]; }
        if (c.nonuniform) {
            q.cells = choose_cells(p, q.inv_2alpha);
            q.cell_scale = std::ldexp(static_cast<float>(q.cells), -149);
            if (q.cells == 0 || !std::isfinite(q.inv_2alpha)) search = kLogGrid;
        }
    }
    if (search == kLogGrid)                                  // one form for the launch
        for (uint32_t i = 0; i < c.n_workers; ++i)
            if ((args.q[i].log_cells = choose_log_grid(c.params[i], &args.q[i].log_base)) == 0) search = kBinary;
    // uniform fp32 rows have no per-block set-up worth sharing: one block per tile (30 M x 8, 16 levels: 156 us, in shares 166);
    // bf16 ones, bound by instructions, do better in shares (124 M x 8, 4 levels: 543 us by tiles, 506 in shares)
    const dim3 grid = compress_grid(c.d, c.n_workers, !is_uniform(search) || c.bf16);
    switch (c.bits) {
        case 1: return dispatch<1>(c, args, grid, search);
        case 2: return dispatch<2>(c, args, grid, search);
        case 3: return dispatch<3>(c, args, grid, search);
        default: return dispatch<4>(c, args, grid, search);
    }
}

template <int BITS>
static cudaError_t dispatch_dev(const CompressCall& c, const TilePlan& plan, bool behind) {
    const auto kernel = c.nonuniform ? (c.bf16 ? (behind ? compress_kernel_dev<BITS, true, true, true> : compress_kernel_dev<BITS, true, true, false>)
                                               : compress_kernel_dev<BITS, true, false, false>)
                                     : (c.bf16 ? compress_kernel_dev<BITS, false, true, false> : compress_kernel_dev<BITS, false, false, false>);
    return launch_kernel(kernel, dim3(plan.blocks), kThreads, 0, c.stream, c.grad, c.grad_stride, c.params_dev, round_keys(c.seed),
                         c.first_worker, c.packed, c.words_stride, plan, c.n_workers * plan.segs.n);
}

cudaError_t launch_compress_dev(const CompressCall& c) {
    // bf16 table codebooks: the decision-table kernel first; it serves the rows its window fits and the element-wise
    // kernel (a small grid then: it normally finds nothing left) takes the others
    bool lut = false;
    if (const cudaError_t e = launch_compress_lut(c, &lut)) return e;
    static thread_local TilePlan plan;
    const uint64_t resident = static_cast<uint64_t>(sm_count()) * TQ_COMPRESS_MIN_BLOCKS;
    plan_tiles(&plan, c.segs, c.d, c.n_workers, 32 * kThreads, lut ? resident / TQ_COMPRESS_MIN_BLOCKS : resident);
    if (const uint64_t more = lut ? 1 : ranges_per_block(plan.per_block); more > 1) plan_tiles(&plan, c.segs, c.d, c.n_workers, 32 * kThreads, resident * more);
    if (c.launches) *c.launches = lut ? 2 : 1;
    switch (c.bits) {
        case 1: return dispatch_dev<1>(c, plan, lut);
        case 2: return dispatch_dev<2>(c, plan, lut);
        case 3: return dispatch_dev<3>(c, plan, lut);
        default: return dispatch_dev<4>(c, plan, lut);
    }
}

}  // namespace tq

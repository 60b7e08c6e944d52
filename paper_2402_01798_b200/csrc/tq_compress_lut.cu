// Client side of Algorithm 1 for gradients stored as bf16: truncate (Section 3.1, truncation equation),
// stochastically round onto the codebook (Section 3.1, quantizer equation) and pack, with the part of
// the decision that does not depend on the random draw taken from a table.
//
// A bf16 element has only 2^16 possible values, and for a given quantizer the interval index k and the
// threshold T = rint(p * 2^16) of the rounding decision are functions of that value alone.  Each block
// therefore evaluates the decision once per bit pattern, with the very operations the element-wise
// kernels use (one IEEE operation per step), and stores X + 65535 with X = k * 2^16 + min(T, 2^16).  An
// element then costs one table read, and code = k + [r < T] = floor((X + 65535 - r) / 2^16) for the
// element's 16 random bits r.
//
// The table is indexed by the pattern itself: positive values from entry 0, negative ones from entry 2^15, each up to P_top,
// the smallest bf16 value >= alpha; nothing is stored between P_top and 2^15.  A packed maximum with -P_top and a packed
// minimum with P_top bring every value into the table, both halves of a word in one operation each; the maximum
// returns the operand that is a number, so a NaN becomes -alpha as in the element-wise form.  Values so small that the
// decision equals that of zero (the host or the block checks this by evaluating the decision at +-base; it is monotone in
// the value) are filled in, not evaluated.
//
// What bounds it: table reads.  32 random words take 3.6 wavefronts of the shared-memory pipe, with the loads 4.3 per 32 elements, 17.2 of
// the 18.5 cycles that the SM's four schedulers take for 32 elements each (a copy's bandwidth would leave 13).  The
// multiplier pipe is busy for 14.9 of them, the integer / compare pipe for 10.2, and the wide multiplies of Philox hold the
// latter up further, so the index and the comparison with r are given to neither more than needed: the two-way dot product of 16-bit
// halves (one operation of the multiplier pipe, 2 cycles) makes the address, table + 4 * pattern, from either half of a word, and
// X + 65535 - r from either half of a word of random bits.  The code is then byte 2 of the difference, and codes are packed by
// byte permutes.  124 M x 8, 16 levels, against an index of clamped binades with the sign moved beside it and r made into a
// float by a byte permute (14.3 instructions per element, now 12.2; integer pipe 14.8 cycles): 601 -> 508 us through device
// parameters, 591 -> 497 with the host's; 4 levels 600 -> 504.
#include <cmath>
#include <type_traits>

#include "tq_device.cuh"
#include "tq_launch.h"
#include "tq_lut.cuh"

namespace tq {

struct LutWorker {
    float alpha;
    uint32_t top, base;   // the largest pattern, the smallest one that is evaluated (without lut_lift of alpha's pattern)
    float levels[TQ_MAX_LEVELS];
    float inv_width[TQ_MAX_LEVELS];
};
struct LutArgs {
    LutWorker q[TQ_MAX_WORKERS];
};

// ---- device ------------------------------------------------------------------------------------------

__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r; asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r;
}
__device__ __forceinline__ uint32_t min_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r; asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r;
}

__device__ __forceinline__ uint32_t mul_bf16x2(uint32_t a, uint32_t b) {
    uint32_t r; asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r;
}

struct LutCtx {
    uint32_t table;          // shared-memory address of entry 0
    uint32_t negtop2, top2;  // the bf16 values -P_top and P_top in both halves
    PhiloxRun pr;
    uint32_t factor2;        // LIFT: 1 or 2^-64 in both halves
};

__device__ __forceinline__ uint32_t lds_u32(uint32_t addr) {
    uint32_t v; asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(addr)); return v;
}

// Elements a thread quantizes as one piece: consecutive, loaded with 256-bit loads (lane after lane, so a
// warp's load covers one contiguous kilobyte), and packing to whole 32-bit words.
template <int BITS> struct Piece { static constexpr int kElems = (BITS == 2 || BITS == 4) ? 16 : 32; };

// One piece whose words are in registers: quantize, pack, store.  LIFT = alpha may be 2^69 or more (see lut_lift).  TAIL = the row's last piece,
// possibly partial.
template <int BITS, bool LIFT, bool TAIL>
__device__ __forceinline__ void lut_piece(const uint32_t (&g)[Piece<BITS>::kElems / 2], uint32_t* prow, uint64_t piece, uint64_t d,
                                          uint64_t words_out, const RoundKeys& rk, const LutCtx& cx) {
    constexpr int E = Piece<BITS>::kElems, GROUPS = E / 8, WORDS = E * BITS / 32;
    const uint64_t j0 = piece * E;
    const uint32_t blk_lo = static_cast<uint32_t>(j0 >> 3);   // rows of more than 2^35 elements do not come here
    uint32_t chunk[GROUPS];
#pragma unroll
    for (int grp = 0; grp < GROUPS; ++grp) {
        uint32_t rnd[4], v[8];
        philox_block(blk_lo + grp, cx.pr, rk, rnd);           // j0 >> 3 is a multiple of GROUPS: no carry
#pragma unroll
        for (int h = 0; h < 4; ++h) {                          // elements 2h, 2h+1 of the group
            const uint32_t in = LIFT ? mul_bf16x2(g[4 * grp + h], cx.factor2) : g[4 * grp + h];
            const uint32_t w = min_bf16x2(max_bf16x2(in, cx.negtop2), cx.top2);
            v[2 * h] = dot_halves_signed(rnd[h], 0x00FFu, lds_u32(dot_halves(w, 0x0004u, cx.table)));           // X + 65535 - r
            v[2 * h + 1] = dot_halves_signed(rnd[h], 0xFF00u, lds_u32(dot_halves(w, 0x0400u, cx.table)));
            if constexpr (TAIL) {                              // padding bits are zero
                if (j0 + 8 * grp + 2 * h >= d) v[2 * h] = 0u;
                if (j0 + 8 * grp + 2 * h + 1 >= d) v[2 * h + 1] = 0u;
            }
        }
        chunk[grp] = pack_byte2<BITS>(v);
    }

    uint32_t w[WORDS];
    if constexpr (BITS == 4) { w[0] = chunk[0]; w[1] = chunk[1]; }
    if constexpr (BITS == 3) {
        w[0] = chunk[0] | (chunk[1] << 24);
        w[1] = (chunk[1] >> 8) | (chunk[2] << 16);
        w[2] = (chunk[2] >> 16) | (chunk[3] << 8);
    }
    if constexpr (BITS == 2) { w[0] = __byte_perm(chunk[0], chunk[1], 0x5410u); }
    if constexpr (BITS == 1) { w[0] = chunk[0] | (chunk[1] << 8) | (chunk[2] << 16) | (chunk[3] << 24); }

    uint32_t* dst = prow + piece * WORDS;
    if constexpr (!TAIL) {
        if constexpr (BITS == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(w[0], w[1]);
        if constexpr (BITS == 3) { dst[0] = w[0]; dst[1] = w[1]; dst[2] = w[2]; }
        if constexpr (BITS == 2 || BITS == 1) dst[0] = w[0];
    } else {
        const uint64_t first = piece * WORDS;
#pragma unroll
        for (int i = 0; i < WORDS; ++i)
            if (first + i < words_out) dst[i] = w[i];
        for (uint64_t k = first + WORDS; k < words_out; ++k) prow[k] = 0u;
    }
}

template <int BITS>
__device__ __forceinline__ void load_piece(const char* row, uint64_t piece, uint32_t (&g)[Piece<BITS>::kElems / 2]) {
    constexpr int E = Piece<BITS>::kElems;
#pragma unroll
    for (int i = 0; i < E / 16; ++i)
        asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=r"(g[8 * i]), "=r"(g[8 * i + 1]), "=r"(g[8 * i + 2]), "=r"(g[8 * i + 3]),
                       "=r"(g[8 * i + 4]), "=r"(g[8 * i + 5]), "=r"(g[8 * i + 6]), "=r"(g[8 * i + 7])
                     : "l"(row + piece * (2 * E) + 32 * i));
}

// One block per SM, with the table that all its warps share.  Codes of 2 and 4 bits, pieces of 16 elements: 24 warps of 80 registers, of which the
// next iteration's loads take 16 while the present one is quantized (124 M x 8, 16 levels, host / device parameters: 497 / 508 us; without them
// 24 warps 547 / 537, 28 warps 518 / 528, 32 warps 539 / 515).  Codes of 1 and 3 bits, pieces of 32: more warps instead (28 warps 500 us, 32 warps
// 535, 24 with the second set 555 and spills).
template <int BITS> struct LutShape {
    static constexpr bool kTwoBuffers = BITS == 2 || BITS == 4;
    static constexpr int kThreads = kTwoBuffers ? 768 : 896;
};

// A block's share of one row: build the table for quantizer q, then quantize the pieces begin + thread, + stride,
// ... below `end`, and with LAST the row's last one, possibly partial.
template <int BITS, bool WAIT, bool LIFT = false>
__device__ __forceinline__ void lut_block(const LutWorker& q, uint32_t* s_table, const char* __restrict__ row,
                                          uint32_t* __restrict__ prow, uint64_t d, uint64_t words_out, uint32_t worker,
                                          const RoundKeys& rk, uint64_t begin, uint64_t stride, uint64_t end, bool last, std::bool_constant<LIFT> = {}) {
    constexpr int kLutThreads = LutShape<BITS>::kThreads;
    const uint32_t lift = LIFT ? lut_lift(top_pattern(q.alpha)) : 0u;
    {
        const LutRule rule{q.alpha, 1u << BITS, q.levels, q.inv_width};
        const uint32_t first = q.base & ~3u, n = q.top + 1 - first;             // everything below `first` is decided like zero
        const uint32_t x0 = decision_x(0.0f, rule) + 65535u;
        for (uint32_t i = threadIdx.x; i < first / 2; i += kLutThreads) {       // four entries at a time, both signs
            const uint32_t at = i < first / 4 ? 4 * i : 0x8000u + 4 * i - first;
            *reinterpret_cast<uint4*>(s_table + at) = make_uint4(x0, x0, x0, x0);
        }
        for (uint32_t i = threadIdx.x; i < 2 * n; i += kLutThreads) {
            const uint32_t pattern = first + (i >= n ? i - n + 0x8000u : i);
            s_table[pattern] = decision_x(bf16_pattern_value(pattern + lift), rule) + 65535u;
        }
    }
    __syncthreads();
    if constexpr (WAIT) pdl_wait();          // the table came from kernel parameters

    constexpr int E = Piece<BITS>::kElems, PER_ITER = 32 / E;   // 32 elements per thread and iteration: four Philox blocks in flight
    const LutCtx cx{smem_addr(s_table), (q.top | 0x8000u) * 0x00010001u, q.top * 0x00010001u, philox_run(0u, worker, rk), lift ? 0x1F801F80u : 0x3F803F80u};
    const uint64_t row_interior = (d - 1) / E, interior = end < row_interior ? end : row_interior;      // whole pieces before the row's last one

    uint64_t piece = begin + threadIdx.x;
    auto fetch = [&](uint32_t (&buf)[PER_ITER][E / 2], uint64_t first) {
#pragma unroll
        for (int k = 0; k < PER_ITER; ++k)
            if (first + k * stride < interior) load_piece<BITS>(row, first + k * stride, buf[k]);
    };
    auto quantize = [&](const uint32_t (&buf)[PER_ITER][E / 2], uint64_t first) {
#pragma unroll
        for (int k = 0; k < PER_ITER; ++k)
            if (first + k * stride < interior) lut_piece<BITS, LIFT, false>(buf[k], prow, first + k * stride, d, words_out, rk, cx);
    };
    uint32_t a[PER_ITER][E / 2];
    if constexpr (LutShape<BITS>::kTwoBuffers) {       // two sets of registers take turns: the next iteration's loads are in flight while this one is quantized
        uint32_t b[PER_ITER][E / 2];
        fetch(a, piece);
        while (piece < interior) {
            const uint64_t next = piece + PER_ITER * stride;
            fetch(b, next);
            quantize(a, piece);
            if (next >= interior) break;
            piece = next + PER_ITER * stride;
            fetch(a, piece);
            quantize(b, next);
        }
    } else {
        for (; piece < interior; piece += PER_ITER * stride) {
            fetch(a, piece);
            quantize(a, piece);
        }
    }
    if (last && threadIdx.x == 0) {
        const unsigned short* e = reinterpret_cast<const unsigned short*>(row);
        uint32_t t[E / 2];
#pragma unroll
        for (int i = 0; i < E / 2; ++i) {
            const uint64_t j = row_interior * E + 2 * i;
            const uint32_t lo = j < d ? ldg16(e + j) : 0u, hi = j + 1 < d ? ldg16(e + j + 1) : 0u;
            t[i] = lo | (hi << 16);
        }
        lut_piece<BITS, LIFT, true>(t, prow, row_interior, d, words_out, rk, cx);
    }
}

// Quantizers passed by value (host-side tq_params); the host has chosen the window.  LIFT: for calls with at least one such row.
template <int BITS, bool LIFT>
__global__ void __launch_bounds__(LutShape<BITS>::kThreads, 1)
compress_lut_kernel(const void* __restrict__ grad, uint64_t d, uint64_t grad_stride, const __grid_constant__ LutArgs args,
                    const __grid_constant__ RoundKeys rk, uint32_t first_worker,
                    uint32_t* __restrict__ packed, uint64_t words_stride, uint64_t words_out) {
    constexpr int kLutThreads = LutShape<BITS>::kThreads;
    extern __shared__ __align__(16) uint32_t s_table[];       // lut_bytes of the largest of the workers' last patterns
    const uint32_t wi = blockIdx.y;
    lut_block<BITS, true>(args.q[wi], s_table, static_cast<const char*>(grad) + static_cast<uint64_t>(wi) * grad_stride * 2,
                    packed + static_cast<uint64_t>(wi) * words_stride, d, words_out, first_worker + wi, rk,
                    static_cast<uint64_t>(blockIdx.x) * kLutThreads, static_cast<uint64_t>(gridDim.x) * kLutThreads, ~0ull, blockIdx.x == 0, std::bool_constant<LIFT>{});
}

// Quantizers read from device memory (tq_params_device).  Every block decides by lut_serves_record whether the
// table form serves its row, with the largest window; rows it does not serve are left to the element-wise
// device-parameter kernels, which are launched after this one and skip the rows served here.
struct LutState {
    LutWorker q;
    uint32_t fits[2];                                         // bit b of the 64: a window of b + 1 binades serves the row
};
// The record's quantizer into s.q; says whether the table serves it.  Block-uniform; ends with a barrier.
template <int BITS>
__device__ __forceinline__ bool lut_record(const tq_params_t& rec, LutState& s) {
    if (threadIdx.x < TQ_MAX_LEVELS) {
        s.q.levels[threadIdx.x] = rec.levels[threadIdx.x];
        s.q.inv_width[threadIdx.x] = rec.inv_width[threadIdx.x];
    }
    const float alpha = rec.alpha;                            // read beside the levels: after a barrier it would be one more trip to memory
    const bool usable = lut_usable(rec, BITS);
    __syncthreads();
    if (!usable) return false;
    const uint32_t top = top_pattern(alpha);
    uint32_t base = 0;
    if (threadIdx.x < kLutBinades) {
        const bool fits = lut_window_fits(LutRule{alpha, 1u << BITS, s.q.levels, s.q.inv_width}, top, kLutBinade * (threadIdx.x + 1), &base);
        const uint32_t bits = __ballot_sync(0xFFFFFFFFu, fits);
        if ((threadIdx.x & 31u) == 0) s.fits[threadIdx.x >> 5] = bits;
    }
    __syncthreads();
    if (s.fits[1] >> 31 == 0) return false;                   // the rule of lut_serves_record: not even the largest window
    const uint32_t n = kLutBinade * (s.fits[0] ? __ffs(static_cast<int>(s.fits[0])) : 32 + __ffs(static_cast<int>(s.fits[1])));
    if (threadIdx.x == 0) {
        s.q.alpha = alpha;
        s.q.top = top;
        s.q.base = top >= n ? top - (n - 1) : 0u;
    }
    __syncthreads();
    return true;
}

template <int BITS>
__global__ void __launch_bounds__(LutShape<BITS>::kThreads, 1)
compress_lut_kernel_dev(const void* __restrict__ grad, uint64_t d, uint64_t grad_stride, const tq_params_t* params,
                        const __grid_constant__ RoundKeys rk, uint32_t first_worker, uint32_t* __restrict__ packed,
                        uint64_t words_stride, uint64_t words_out) {
    extern __shared__ __align__(16) uint32_t s_table[];       // kLutMostBytes
    constexpr int kLutThreads = LutShape<BITS>::kThreads;
    __shared__ LutState s;
    const uint32_t wi = blockIdx.y;
    pdl_wait();
    if (!lut_record<BITS>(params[wi], s)) return;
    lut_block<BITS, false>(s.q, s_table, static_cast<const char*>(grad) + static_cast<uint64_t>(wi) * grad_stride * 2,
                    packed + static_cast<uint64_t>(wi) * words_stride, d, words_out, first_worker + wi, rk,
                    static_cast<uint64_t>(blockIdx.x) * kLutThreads, static_cast<uint64_t>(gridDim.x) * kLutThreads, ~0ull, blockIdx.x == 0);
}

// Layer groups: a block's range of the jobs' tiles (kLutThreads pieces each), a table for every piece of a job.
template <int BITS>
__global__ void __launch_bounds__(LutShape<BITS>::kThreads, 1)
compress_lut_kernel_segs(const void* __restrict__ grad, uint64_t grad_stride, const tq_params_t* params,
                         const __grid_constant__ RoundKeys rk, uint32_t first_worker, uint32_t* __restrict__ packed, uint64_t words_stride,
                         const __grid_constant__ TilePlan plan, uint32_t start_tiles) {
    extern __shared__ __align__(16) uint32_t s_table[];       // kLutMostBytes
    constexpr int kLutThreads = LutShape<BITS>::kThreads;
    __shared__ LutState s;
    uint64_t cur = first_tile_of_block(plan, blockIdx.x);
    const uint64_t range_end = first_tile_of_block(plan, blockIdx.x + 1);
    pdl_wait();
    while (cur < range_end) {
        JobPiece job = next_piece(plan, cur, range_end);
        if (job.tile1 <= start_tiles) continue;                // nothing of the job itself
        job.tile0 = job.tile0 > start_tiles ? job.tile0 - start_tiles : 0;
        job.tile1 -= start_tiles;
        if (lut_record<BITS>(params[job.job], s))
            lut_block<BITS, false>(s.q, s_table,
                                   static_cast<const char*>(grad) + (static_cast<uint64_t>(job.worker) * grad_stride + job.off) * 2,
                                   packed + static_cast<uint64_t>(job.worker) * words_stride + plan.segs.woff[job.seg], job.d,
                                   (((job.d * BITS + 31) >> 5) + 3) & ~static_cast<uint64_t>(3), first_worker + job.worker, rk,
                                   job.tile0 * kLutThreads, kLutThreads, job.tile1 * kLutThreads, job.last);
        __syncthreads();                                       // the next piece reuses the table
    }
}

// ---- host --------------------------------------------------------------------------------------------

constexpr int lut_bytes(uint32_t top) { return static_cast<int>((0x8000u + top + 1) * sizeof(uint32_t)); }
constexpr int kLutMostBytes = lut_bytes(kLutMostTop);

// First pattern that has to be evaluated; false if no window of at most kLutBinades binades serves the quantizer.
static bool first_pattern(const LutRule& q, uint32_t top, uint32_t* base) {
    // a window that fits stays valid when it is made larger: halve the range of sizes
    uint32_t lo = 0, hi = kLutBinades;
    if (!lut_window_fits(q, top, hi * kLutBinade, base)) return false;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) / 2;
        if (lut_window_fits(q, top, mid * kLutBinade, base)) hi = mid; else lo = mid;
    }
    return lut_window_fits(q, top, hi * kLutBinade, base);
}

template <int BITS, bool LIFT>
static cudaError_t launch_lut_form(const CompressCall& c, const LutArgs& args, uint32_t top, uint32_t per_worker) {
    // always the same limit: another thread may set it between this call's and the launch
    const cudaError_t e = cudaFuncSetAttribute(compress_lut_kernel<BITS, LIFT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLutMostBytes);
    if (e != cudaSuccess) return e;
    return launch_kernel(compress_lut_kernel<BITS, LIFT>, dim3(per_worker, c.n_workers), LutShape<BITS>::kThreads, lut_bytes(top), c.stream, c.grad, c.d,
                         c.grad_stride, args, round_keys(c.seed), c.first_worker, c.packed, c.words_stride, c.words_out);
}
template <int BITS>
static cudaError_t launch_lut(const CompressCall& c, const LutArgs& args, uint32_t top, uint32_t per_worker, bool lift) {
    return lift ? launch_lut_form<BITS, true>(c, args, top, per_worker) : launch_lut_form<BITS, false>(c, args, top, per_worker);
}

// Blocks per row, and what the longest chain of blocks costs with them, in elements that a block quantizes in that time.  The waves follow one
// another, each with its tables: 30 M x 1 in 1 / 2 / 3 / 4 / 8 waves 19.0 / 22.9 / 26.7 / 30.6 / 45.2 us with 16 levels, 19.0 / 21.2 / 24.6 / 27.8 / 40.9
// with 8, 3.8 and 3.1 us a table or 50000 and 40000 elements.  Rows that do not divide the SMs waste less in several waves (124 M x 8, 16 levels,
// 18 / 36 / 37 / 55 / 74 blocks a row: 527 / 531 / 518 / 527 / 527 us; 25.6 M x 16, 9 / 18 / 27 / 37 / 46: 212 / 217 / 221 / 220 / 226).  With codes of 1
// and 3 bits more and shorter shares also even out SMs of different speed, 3 % of a share, at the largest sizes (8 levels, 193 M x 2 in 1 / 2 waves
// 250 / 232 us, 46 M x 11 in 1 / 3 317 / 306); with 2 and 4 bits they do not (16 levels 210 / 210 and 280 / 280).
static uint64_t lut_plan(const CompressCall& c, uint32_t* per_worker) {
    const bool two_buffers = c.bits % 2 == 0;
    const uint64_t d = c.d, n_workers = c.n_workers, table = two_buffers ? 50000 : 40000;
    const uint64_t sms = static_cast<uint64_t>(sm_count());
    uint64_t best = ~0ull;
    for (uint64_t shares = 1; shares <= 8; ++shares) {
        uint64_t p = sms * shares / n_workers;
        if (p == 0) p = 1;
        const uint64_t waves = (p * n_workers + sms - 1) / sms, share = d / p + 1;
        const uint64_t cost = waves * (table + share) + (two_buffers ? 0 : share / 32);
        if (cost < best) { best = cost; *per_worker = static_cast<uint32_t>(p); }
    }
    return best;
}

template <int BITS>
static cudaError_t launch_lut_dev(const CompressCall& c, uint32_t per_worker) {
    cudaError_t e = cudaFuncSetAttribute(compress_lut_kernel_dev<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLutMostBytes);
    if (e != cudaSuccess) return e;
    return launch_kernel(compress_lut_kernel_dev<BITS>, dim3(per_worker, c.n_workers), LutShape<BITS>::kThreads, kLutMostBytes, c.stream, c.grad,
                         c.d, c.grad_stride, c.params_dev, round_keys(c.seed), c.first_worker, c.packed, c.words_stride, c.words_out);
}

// One range per SM.  The start of a job within a range -- its record, its table, its last piece, the loads' first latency -- takes as long as 80000
// elements and is counted with the tiles, or a range of many short jobs holds up all others (16 levels, groups of lengths up to 75 apart, started
// for nothing / as 40000 / 80000 / 160000 elements: 25.6 M x 16 in 16 groups 291 / 274 / 264 / 267 us, 10 M x 8 in 16 92 / 72 / 65 / 68, 124 M x 8 in 16
// 581 / 566 / 558 / 559; two ranges per SM 269, 71 and 564 at best).
constexpr uint64_t kLutStartElems = 80000;
template <int BITS>
static cudaError_t launch_lut_segs(const CompressCall& c, uint32_t blocks) {
    static thread_local TilePlan plan;
    constexpr uint64_t tile = static_cast<uint64_t>(LutShape<BITS>::kThreads) * Piece<BITS>::kElems;
    constexpr uint32_t start_tiles = static_cast<uint32_t>((kLutStartElems + tile / 2) / tile);
    plan_tiles(&plan, c.segs, c.d, c.n_workers, tile, blocks, start_tiles);
    const cudaError_t e = cudaFuncSetAttribute(compress_lut_kernel_segs<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLutMostBytes);
    if (e != cudaSuccess) return e;
    return launch_kernel(compress_lut_kernel_segs<BITS>, dim3(plan.blocks), LutShape<BITS>::kThreads, kLutMostBytes, c.stream, c.grad, c.grad_stride, c.params_dev,
                         round_keys(c.seed), c.first_worker, c.packed, c.words_stride, plan, start_tiles);
}

// The element-wise kernels take about 1.7 times as long per element and build no table.  With host parameters the line is higher than that, because
// behind another kernel the table is built early; with device parameters lower, because there it is not and a second launch looks for rows
// that the table does not serve.  In both cases from about 8 M (12 M) elements that divide the SMs evenly.  Table / element-wise, 16 levels, host
// and device parameters: 8 M 7.5 / 9.6 and 11.3 / 11.4 us, 12.5 M 9.8 / 12.7 and 13.3 / 15.7, 2 M x 8 11.8 / 17.5 and 16.2 / 19.3, 250 k x 64 (128
// blocks for 148 SMs) 18.4 / 20.1 with device parameters, 24 M 15.4 / 22.1 and 19.2 / 23.9, 124 M x 8 501 / 843 and 508 / 843.  Codes of 1 and 3
// bits with host parameters from 1.65 on where a thread has more than two of their long pieces: such parameters often come to an idle GPU (the
// records have just been waited for), where nothing hides the table.  Call and wait on an idle GPU, 8 levels, table / element-wise: 8 M 19.5 / 20.3 us,
// 9 M 21.5 / 20.4, 562500 x 16 24.3 / 21.9, 10 M 21.6 / 21.8, 625 k x 16 24.0 / 25.5; 16 levels 9 M 19.5 / 21.5, 562500 x 16 23.0 / 23.0.
static bool lut_pays(const CompressCall& c, uint32_t* per_worker) {
    const uint64_t cost = lut_plan(c, per_worker), others = c.d * c.n_workers / static_cast<uint64_t>(sm_count());
    if (c.bits % 2 == 0) return cost * 100 < others * (c.params_dev ? 162 : 194);
    const bool late = c.d / *per_worker > 2ull * LutShape<3>::kThreads * Piece<3>::kElems;      // 1 and 3 bits: the same shape
    return cost * 100 < others * (c.params_dev ? 153 : late ? 165 : 178);
}

cudaError_t launch_compress_lut(const CompressCall& c, bool* applied) {
    *applied = false;
    uint32_t per_worker = 0;
    if (!c.bf16 || !c.nonuniform) return cudaSuccess;
    if (c.segs) {
        uint64_t total = 0;
        for (uint32_t s = 0; s < c.segs->n; ++s) {
            if (c.segs->len[s] > (1ull << 35)) return cudaSuccess;
            total += c.segs->len[s] * c.n_workers;
        }
        // The start of a piece against what the table saves; the element-wise kernel as above.  Table / element-wise, 16 levels, groups of lengths up to 75
        // apart: 25.6 M x 16 in 16 264 / 361 us, 10 M x 8 in 16 65 / 80, 2 M x 64 in 5 107 / 123, 4 M x 8 in 5 29 / 34, 10 M x 8 in 40 83 / 82.
        const uint32_t blocks = static_cast<uint32_t>(sm_count());
        if ((blocks + static_cast<uint64_t>(c.n_workers) * c.segs->n) * kLutStartElems * 100 >= total * 48) return cudaSuccess;
        *applied = true;
        switch (c.bits) {
            case 1: return launch_lut_segs<1>(c, blocks);
            case 2: return launch_lut_segs<2>(c, blocks);
            case 3: return launch_lut_segs<3>(c, blocks);
            default: return launch_lut_segs<4>(c, blocks);
        }
    }
    if (c.d > (1ull << 35) || !lut_pays(c, &per_worker)) return cudaSuccess;
    if (c.params_dev) {      // the kernel decides row by row; the caller launches the element-wise kernels for the rest
        *applied = true;
        switch (c.bits) {
            case 1: return launch_lut_dev<1>(c, per_worker);
            case 2: return launch_lut_dev<2>(c, per_worker);
            case 3: return launch_lut_dev<3>(c, per_worker);
            default: return launch_lut_dev<4>(c, per_worker);
        }
    }
    static thread_local LutArgs args;
    uint32_t most = 0;
    bool lift = false;
    for (uint32_t i = 0; i < c.n_workers; ++i) {
        const tq_params_t& p = c.params[i];
        if (!(p.alpha > 0.0f) || !(p.alpha <= 3.402823466e38f)) return cudaSuccess;
        LutWorker& q = args.q[i];
        q.top = top_pattern(p.alpha);
        if (!first_pattern(lut_rule(p, c.bits), q.top, &q.base)) return cudaSuccess;
        const uint32_t low = lut_lift(q.top);
        lift = lift || low != 0;
        q.top -= low;
        q.base -= low;
        most = q.top > most ? q.top : most;
        q.alpha = p.alpha;
        for (int k = 0; k < TQ_MAX_LEVELS; ++k) { q.levels[k] = p.levels[k]; q.inv_width[k] = p.inv_width[k]; }
    }
    *applied = true;
    switch (c.bits) {
        case 1: return launch_lut<1>(c, args, most, per_worker, lift);
        case 2: return launch_lut<2>(c, args, most, per_worker, lift);
        case 3: return launch_lut<3>(c, args, most, per_worker, lift);
        default: return launch_lut<4>(c, args, most, per_worker, lift);
    }
}

}  // namespace tq

// Device-side building blocks shared by the libtq kernels (sm_100a).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "tq.h"
#include "tq_launch.h"

namespace tq {

constexpr int kThreads = 256;
constexpr float kMagic = 8388608.0f;          // 2^23: adding it leaves an integer in the mantissa
constexpr uint32_t kMagicBits = 0x4B000000u;  // bit pattern of 2^23

// The kernel before this one on the stream is complete and its writes are visible; the next one may be set up.  Nothing
// before this may touch global memory, and nothing may let the compiler move a load up to there: what other kernels write is read
// through volatile asm, or through pointers that make no promise (const together with __restrict__, like __ldg, says that the
// data does not change while the kernel runs, and an early start begins while it still does).
__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
}

// ---- 256-bit global accesses (one full 32-byte sector per lane) ---------------------------------
__device__ __forceinline__ void ldg256_stream(const void* p, uint32_t (&v)[8]) {
    asm volatile("ld.global.nc.L1::no_allocate.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
                 : "l"(p));
}
__device__ __forceinline__ void ldg256(const float* p, float (&v)[8]) {
    asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p) : "memory");
}
__device__ __forceinline__ void stg256(void* p, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%8], {%0,%1,%2,%3,%4,%5,%6,%7};"
                 :: "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]), "l"(p)
                 : "memory");
}

// Eight consecutive gradient elements kept as loaded (fp32: 8 words; bf16: 4 words of two), decoded
// on use.  Keeping bf16 packed halves the registers a loaded group occupies.  The address is 32-byte aligned for fp32 and 16-byte
// aligned for bf16.  bf16 -> fp32 is exact: the stored 16 bits become the high half of the fp32 pattern.
template <bool BF16>
struct Raw8 {
    uint32_t v[BF16 ? 4 : 8];
};
template <bool BF16>
__device__ __forceinline__ void load8_raw(const void* p, Raw8<BF16>& r) {
    if constexpr (!BF16) ldg256_stream(p, r.v);
    else asm volatile("ld.global.nc.L1::no_allocate.v4.b32 {%0,%1,%2,%3}, [%4];"
                      : "=r"(r.v[0]), "=r"(r.v[1]), "=r"(r.v[2]), "=r"(r.v[3]) : "l"(p));
}
template <bool BF16>
__device__ __forceinline__ float elem(const Raw8<BF16>& r, int e) {
    if constexpr (!BF16) return __uint_as_float(r.v[e]);
    else return __uint_as_float((e & 1) ? (r.v[e >> 1] & 0xFFFF0000u) : (r.v[e >> 1] << 16));
}

// Single words, any alignment of the run they belong to.
__device__ __forceinline__ uint32_t ldg32(const void* p) {
    uint32_t v; asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(p)); return v;
}
__device__ __forceinline__ uint32_t ldg16(const void* p) {
    unsigned short v; asm volatile("ld.global.nc.b16 %0, [%1];" : "=h"(v) : "l"(p)); return v;
}
// One element, any alignment (ragged tails).
template <bool BF16>
__device__ __forceinline__ float load1(const void* base, uint64_t j) {
    if constexpr (!BF16) return __uint_as_float(ldg32(static_cast<const float*>(base) + j));
    else return __uint_as_float(ldg16(static_cast<const unsigned short*>(base) + j) << 16);
}

// ---- asynchronous copies into shared memory, counted on an mbarrier ----------------------------------
// Every wait is bounded: after kWaitLimit polls the caller gets `false`, records it and winds down.
constexpr uint32_t kWaitLimit = 1u << 22;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// global -> this block's shared memory, `bytes` a multiple of 16, both addresses 16-byte aligned
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t it = 0; it < kWaitLimit; ++it) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}


// ---- packed fp32 pairs ----------------------------------------------------------------------------
// sm_100 executes add / mul / fma on two fp32 values held in a 64-bit register pair as ONE instruction,
// each half rounded exactly like the scalar operation.  The kernels here are bound by instruction
// issue, so pairing halves the cost of every arithmetic step it applies to.
struct f32x2 { uint64_t v; };
__device__ __forceinline__ f32x2 pair(float lo, float hi) {
    f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi)); return r;
}
__device__ __forceinline__ f32x2 both(float x) { return pair(x, x); }
__device__ __forceinline__ void unpair(f32x2 p, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p.v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f32x2 add2_rd(f32x2 a, f32x2 b) {   // round toward -infinity
    f32x2 r; asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f32x2 mul2_rd(f32x2 a, f32x2 b) {
    f32x2 r; asm("mul.rm.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v)); return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v)); return r;
}

// ---- Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), counter = (c0, c1, worker, 0) ------------------
// The ten round keys (key advanced by the Weyl constants) are computed once on the host: they depend on
// the seed only, and sit in the kernel's constant bank instead of registers.
struct RoundKeys {
    uint32_t k0[10], k1[10];
};
inline RoundKeys round_keys(uint64_t seed) {
    RoundKeys rk;
    uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
    for (int r = 0; r < 10; ++r) { rk.k0[r] = k0; rk.k1[r] = k1; k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    return rk;
}

__device__ __forceinline__ void mul_wide(uint32_t a, uint32_t b, uint32_t& hi, uint32_t& lo) {
    uint64_t p;
    asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
    asm("mov.b64 {%0, %1}, %2;" : "=r"(lo), "=r"(hi) : "l"(p));
}

// Within a run of elements only c0 changes, so what the first two rounds make of the other three counter
// words is computed once per run: of the 20 wide multiplies of a block, 3 drop out (the second product of
// round 1 and the first of round 2 have constant operands, and word 0 after round 1 is constant).
struct PhiloxRun {
    uint32_t a1, b1, b2, d2;
};
__device__ __forceinline__ PhiloxRun philox_run(uint32_t c1, uint32_t worker, const RoundKeys& rk) {
    uint32_t hi1, lo1;
    mul_wide(0xCD9E8D57u, worker, hi1, lo1);                  // round 1, second product
    const uint32_t c0_1 = hi1 ^ c1 ^ rk.k0[0];                // word 0 after round 1
    uint32_t hi0c, lo0c;
    mul_wide(0xD2511F53u, c0_1, hi0c, lo0c);                  // round 2, first product
    PhiloxRun r;
    r.a1 = rk.k1[0];                 // word 2 after round 1 = hi(M0 * c0) ^ 0 ^ k1[0]
    r.b1 = lo1 ^ rk.k0[1];           // word 0 after round 2 = hi(M1 * word 2) ^ lo1 ^ k0[1]
    r.b2 = hi0c ^ rk.k1[1];          // word 2 after round 2 = hi0c ^ lo(M0 * c0) ^ k1[1]
    r.d2 = lo0c;                     // word 3 after round 2
    return r;
}
__device__ __forceinline__ void philox_block(uint32_t c0, const PhiloxRun& pr, const RoundKeys& rk, uint32_t (&out)[4]) {
    uint32_t hi0, lo0, hi1, lo1;
    mul_wide(0xD2511F53u, c0, hi0, lo0);                      // round 1
    const uint32_t w2 = hi0 ^ pr.a1;
    mul_wide(0xCD9E8D57u, w2, hi1, lo1);                      // round 2
    uint32_t x0 = hi1 ^ pr.b1, x1 = lo1, x2 = lo0 ^ pr.b2, x3 = pr.d2;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        mul_wide(0xD2511F53u, x0, hi0, lo0);
        mul_wide(0xCD9E8D57u, x2, hi1, lo1);
        x0 = hi1 ^ x1 ^ rk.k0[r];
        x2 = hi0 ^ x3 ^ rk.k1[r];
        x1 = lo1;
        x3 = lo0;
    }
    out[0] = x0; out[1] = x1; out[2] = x2; out[3] = x3;
}

// ---- 16-bit halves and packing ------------------------------------------------------------------------
// c + a.lo * w.byte0 + a.hi * w.byte1: the halves of a without sign, the bytes of w without / with.  One operation of the
// multiplier pipe, 2 cycles, where a shift or a mask and an addition are two of the integer / compare pipe, 2 cycles each.
__device__ __forceinline__ uint32_t dot_halves(uint32_t a, uint32_t w, uint32_t c) {
    uint32_t r; asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(w), "r"(c)); return r;
}
__device__ __forceinline__ uint32_t dot_halves_signed(uint32_t a, uint32_t w, uint32_t c) {
    uint32_t r; asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(w), "r"(c)); return r;
}
// The codes in byte 2 of eight words -> their 8 * BITS packed bits, LSB first.
template <int BITS>
__device__ __forceinline__ uint32_t pack_byte2(const uint32_t (&v)[8]) {
    auto four = [](uint32_t a, uint32_t b, uint32_t c, uint32_t d) {       // byte 2 of each
        return __byte_perm(__byte_perm(a, b, 0x0062u), __byte_perm(c, d, 0x0062u), 0x5410u);
    };
    if constexpr (BITS <= 2) {
        // c0 .. c3 side by side in the top byte of a product; the other partial products are disjoint bits below it
        constexpr uint32_t K = (1u << 24) + (1u << (16 + BITS)) + (1u << (8 + 2 * BITS)) + (1u << (3 * BITS));
        const uint32_t lo = four(v[0], v[1], v[2], v[3]) * K, hi = four(v[4], v[5], v[6], v[7]) * K;
        if constexpr (BITS == 2) return __byte_perm(lo, hi, 0x0073u);      // 16 bits; the callers merge chunks by byte permutes
        else return (lo >> 24) | ((hi >> 24) << 4);
    } else {
        const uint32_t t = four(v[0], v[2], v[4], v[6]) + (four(v[1], v[3], v[5], v[7]) << BITS);      // two codes per byte
        if constexpr (BITS == 4) return t;
        const uint32_t u = (t & 0x003F003Fu) | ((t >> 2) & 0x0FC00FC0u);                                // four codes per half
        return (u & 0xFFFu) | ((u >> 4) & 0xFFF000u);
    }
}

// ---- a block's pieces (see TilePlan) ---------------------------------------------------------------
struct JobPiece {
    uint32_t worker, seg, job;
    uint64_t tile0, tile1;         // the piece's tiles, counted from the job's first
    uint64_t d, off;               // the job's elements, and where they start in the worker's row
    bool last;                     // the piece holds the job's last tile
};
__device__ __forceinline__ uint64_t first_tile_of_block(const TilePlan& plan, uint32_t b) {
    return b * plan.per_block + b * plan.rest / plan.blocks;           // b * rest < blocks^2 < 2^32
}
__device__ __forceinline__ uint32_t block_of_tile(const TilePlan& plan, uint64_t t) {
    uint32_t b = static_cast<uint32_t>(static_cast<double>(t) * plan.blocks_per_tile);
    while (first_tile_of_block(plan, b) > t) --b;
    while (first_tile_of_block(plan, b + 1) <= t) ++b;
    return b;
}
// The piece that starts at tile `cur` of the range [.., end); cur moves on to the next one.
__device__ __forceinline__ JobPiece next_piece(const TilePlan& plan, uint64_t& cur, uint64_t end) {
    JobPiece p;
    p.worker = static_cast<uint32_t>(static_cast<double>(cur) * plan.rows_per_tile);      // below 2^53: at most one off
    while (p.worker * plan.per_worker > cur) --p.worker;
    while ((p.worker + 1) * plan.per_worker <= cur) ++p.worker;
    const uint64_t row0 = p.worker * plan.per_worker, in_row = cur - row0;
    p.seg = 0;                     // eight at a time first: one after the other, 40 groups cost more than a microsecond a piece
    while (p.seg + 8 < plan.segs.n && plan.begin[p.seg + 8] <= in_row) p.seg += 8;
    while (p.seg + 1 < plan.segs.n && plan.begin[p.seg + 1] <= in_row) ++p.seg;
    p.job = p.worker * plan.segs.n + p.seg;
    const uint64_t job_end = row0 + plan.begin[p.seg + 1], stop = end < job_end ? end : job_end;
    p.tile0 = in_row - plan.begin[p.seg];
    p.tile1 = p.tile0 + (stop - cur);
    p.last = stop == job_end;
    p.d = plan.segs.len[p.seg]; p.off = plan.segs.off[p.seg];
    cur = stop;
    return p;
}
// First and last block that have a piece of the job.
__device__ __forceinline__ void blocks_of_job(const TilePlan& plan, const JobPiece& p, uint32_t& first, uint32_t& last) {
    const uint64_t row0 = p.worker * plan.per_worker;
    first = block_of_tile(plan, row0 + plan.begin[p.seg]);
    last = block_of_tile(plan, row0 + plan.begin[p.seg + 1] - 1);
}

// ---- warp / block reductions -----------------------------------------------------------------------
// lane 0 gets the sum of the first LANES lanes, all when not stated
template <int LANES = 32, class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xFFFFFFFFu, v, o);
    return v;
}
// of values that are not negative: their bit patterns are in the same order
__device__ __forceinline__ float warp_max_abs(float v) { return __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(v))); }

}  // namespace tq

// Statistics reduction feeding the parameter design of Section 4: per worker sum|g|, sum g^2, max|g|,
// the non-finite count, and for the threshold g_min the tail count n = #{|g_j| > g_min} and
// sum ln(|g_j| / g_min) (the two ingredients of the maximum-likelihood tail index of Section 5 and of
// rho, the tail mass of Section 4.1).
//
// Arithmetic: a thread takes chunks of 64 bytes (16 fp32 or 32 bf16 elements), keeps fp32 partial sums inside a
// chunk (at most 16 terms in a row) and fp64 sums across chunks.  A chunk with a NaN or an Inf is redone element by element in
// fp64.  bf16 pairs are summed, squared and compared as they are (packed and mixed-precision instructions); unpacking
// them first cost 4 instructions per pair.
//
// Shapes.  Short rows (stats_small_kernel): a cluster of 8 blocks per job does everything in one launch, with the
// block sums exchanged through distributed shared memory.  Other rows: the tiles (256 chunks) of all jobs -- workers, or
// (worker, segment) pairs -- are cut into contiguous ranges, one per block (StatsPlan); a block writes one record per
// piece of a job, and the next launch starts by folding the records of the jobs it needs, in index order, so
// that the result does not depend on the order in which blocks run and no block waits for another.
//   automatic threshold, g_min = kappa * mean|g|: pass 1 (moments), pass 2 (tail);
//   hinted threshold: one pass for two candidate thresholds, then a launch that finishes the record and reads the data
//   again only for jobs whose hint missed;
//   caller's threshold: one pass, then a launch that folds the records, a block per job.
// HBM traffic per element and pass: 4 bytes (fp32) or 2 bytes (bf16) read.
#include <math_constants.h>

#include <mutex>

#include "tq_device.cuh"
#include "tq_launch.h"

namespace tq {

constexpr int kRecordsPerJob = 1024;          // scratch records per job: a call has at most blocks + jobs pieces
constexpr int kChunkBytes = 64;
template <bool BF16> constexpr int kChunk = kChunkBytes / (BF16 ? 2 : 4);      // elements
constexpr float kMaxFinite = 3.402823466e38f;

struct alignas(64) Partial {                  // warp_fold reads it as eight doubles
    double sum_abs, sum_sq, sum_log2[2];
    unsigned long long n_tail[2], n_bad;
    float max_abs, pad;
};
// scratch layout for n jobs: [n * kRecordsPerJob] Partial (piece of block b and job j: record b + j), then [n][2] tickets (uint32)
__host__ __device__ inline size_t tickets_offset(uint32_t n_jobs) {
    return static_cast<size_t>(n_jobs) * kRecordsPerJob * sizeof(Partial);
}
size_t stats_workspace_bytes(uint32_t n_workers) {
    return tickets_offset(n_workers) + static_cast<size_t>(n_workers) * 2 * sizeof(uint32_t) + 256;
}

// ---- one chunk -----------------------------------------------------------------------------------------

// Hardware base-2 logarithm (absolute error about 2^-22 for arguments near 1, 2 ulp elsewhere).
__device__ __forceinline__ float lg2_fast(float x) {
    float r; asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x)); return r;
}
__device__ __forceinline__ float fma_sat(float a, float b, float c) {
    float r; asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r;
}
// Two bf16 values at a time; the products and sums of the mixed forms are fp32 with one rounding.
__device__ __forceinline__ uint32_t max_b2(uint32_t a, uint32_t b) { uint32_t r; asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b)); return r; }
__device__ __forceinline__ void add_halves(uint32_t w, float& lo, float& hi) {          // lo += w.lo, hi += w.hi
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tadd.rn.f32.bf16 %0, l, %0;\n\tadd.rn.f32.bf16 %1, h, %1;\n\t}" : "+f"(lo), "+f"(hi) : "r"(w));
}
__device__ __forceinline__ void add_squares(uint32_t w, float& lo, float& hi) {         // lo += w.lo^2, hi += w.hi^2
    asm("{\n\t.reg .b16 l, h;\n\tmov.b32 {l, h}, %2;\n\tfma.rn.f32.bf16 %0, l, l, %0;\n\tfma.rn.f32.bf16 %1, h, h, %1;\n\t}" : "+f"(lo), "+f"(hi) : "r"(w));
}

using Words = uint32_t[16];                    // a chunk as loaded
__device__ __forceinline__ void load_chunk(const char* row, uint64_t c, Words& w) {
    uint32_t v[8];
    ldg256_stream(row + c * kChunkBytes, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) w[i] = v[i];
    ldg256_stream(row + c * kChunkBytes + 32, v);
#pragma unroll
    for (int i = 0; i < 8; ++i) w[8 + i] = v[i];
}
// |g| of the chunk (bf16 pairs lose their signs in place; fp32 uses take the absolute value as an operand modifier)
template <bool BF16>
__device__ __forceinline__ void drop_signs(Words& w) {
    if constexpr (BF16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] &= 0x7FFF7FFFu;
    }
}
// fp32 sums of |g| and g^2; their sum is finite exactly when the chunk can be used as it is.
template <bool BF16>
__device__ __forceinline__ void moments(const Words& w, float& s_abs, float& s_sq) {
    if constexpr (BF16) {
        float a[4] = {0.0f, 0.0f, 0.0f, 0.0f}, q[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            add_halves(w[i], a[0], a[1]); add_halves(w[i + 1], a[2], a[3]);
            add_squares(w[i], q[0], q[1]); add_squares(w[i + 1], q[2], q[3]);
        }
        s_abs = (a[0] + a[1]) + (a[2] + a[3]);
        s_sq = (q[0] + q[1]) + (q[2] + q[3]);
    } else {
        s_abs = 0.0f;
        f32x2 q2 = both(0.0f);
#pragma unroll
        for (int i = 0; i < 16; i += 2) {
            const f32x2 x = pair(__uint_as_float(w[i]), __uint_as_float(w[i + 1]));
            s_abs += fabsf(__uint_as_float(w[i]));
            s_abs += fabsf(__uint_as_float(w[i + 1]));
            q2 = fma2(x, x, q2);
        }
        float q0, q1;
        unpair(q2, q0, q1);
        s_sq = q0 + q1;
    }
}
// Running maximum of |g|: an fp32 value, or two bf16 values.
template <bool BF16>
__device__ __forceinline__ uint32_t chunk_max(const Words& w, uint32_t running) {
    if constexpr (BF16) {
#pragma unroll
        for (int i = 0; i < 16; ++i) running = max_b2(running, w[i]);
        return running;
    } else {
        float m = __uint_as_float(running);
#pragma unroll
        for (int i = 0; i < 16; i += 2) m = fmaxf(fmaxf(m, fabsf(__uint_as_float(w[i]))), fabsf(__uint_as_float(w[i + 1])));
        return __float_as_uint(m);
    }
}
template <bool BF16>
__device__ __forceinline__ float max_value(uint32_t running) {
    if constexpr (BF16) return fmaxf(__uint_as_float(running << 16), __uint_as_float(running & 0xFFFF0000u));
    else return __uint_as_float(running);
}

// Tail sums for K thresholds that are powers of two, t and 2 t: s_log[k] = sum of log2|g| over |g| > t_k, cnt[k] its number.
// The integer / compare pipe runs at half rate and would bound this loop (two compares, two selects and two integer
// adds per threshold), so the tail test m = [|g| > t] is done on the multiply-add pipe, as a saturating fma:
//   fp32: r = |g| / t is exact (t a power of two), m = sat(r * 2^30 - 2^30): the smallest r above 1 gives 2^7, r <= 1 gives <= 0,
//         NaN gives 0, Inf gives 1; for 2 t the same r with 2^29;
//   bf16: the values next above and below t differ from it by 0.011 and 0.006 in log2, a thousand times the error of lg2, so
//         m = sat((lg - log2 t) * 2^10 - 5.7) is 0 or 1 as well, and r is not needed.
// Counts are small floats, and the masked sum is s + m * lg, which rounds exactly like adding lg or nothing, so the sums
// of a threshold do not depend on which of the two it is.  log2 is taken of max(|g|, 2^-126) so that a zero cannot turn
// 0 * (-inf) into NaN; elements that small are never in a tail (t >= 2^-126).
struct TailTest {
    float a, c[2];           // fp32: 1 / t, unused; bf16: unused, the constants of the two saturating operations
    __device__ __forceinline__ explicit TailTest(float t) {
        a = __frcp_rn(t);    // exact; 0 for t = Inf (no hint): nothing is in the tail
        const float e = static_cast<float>(static_cast<int>(__float_as_uint(t) >> 23) - 127);
        c[0] = -1024.0f * e - 5.7f;
        c[1] = -1024.0f * e - 1029.7f;
    }
};
template <bool BF16, int K>
__device__ __forceinline__ void tail_pow2(const Words& w, const TailTest& test, float (&s_log)[K], float (&cnt)[K]) {
    f32x2 log2s[K], cnts[K];
#pragma unroll
    for (int k = 0; k < K; ++k) { log2s[k] = both(0.0f); cnts[k] = both(0.0f); }
#pragma unroll
    for (int i = 0; i < 16; i += BF16 ? 1 : 2) {
        float x0, x1, l0, l1;                                 // what the tail test looks at, log2|g|
        if constexpr (BF16) {
            const uint32_t b = max_b2(w[i], 0x00800080u);
            x0 = l0 = lg2_fast(__uint_as_float(b << 16));
            x1 = l1 = lg2_fast(__uint_as_float(b & 0xFFFF0000u));
        } else {
            unpair(mul2(pair(__uint_as_float(w[i]), __uint_as_float(w[i + 1])), both(test.a)), x0, x1);
            l0 = lg2_fast(fmaxf(fabsf(__uint_as_float(w[i])), 1.17549435e-38f));
            l1 = lg2_fast(fmaxf(fabsf(__uint_as_float(w[i + 1])), 1.17549435e-38f));
        }
        const f32x2 lg = pair(l0, l1);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            f32x2 m;
            if constexpr (BF16) m = pair(fma_sat(x0, 1024.0f, test.c[k]), fma_sat(x1, 1024.0f, test.c[k]));
            else {
                const float scale = k ? 536870912.0f : 1073741824.0f;
                m = pair(fma_sat(fabsf(x0), scale, -1073741824.0f), fma_sat(fabsf(x1), scale, -1073741824.0f));
            }
            log2s[k] = fma2(m, lg, log2s[k]);
            cnts[k] = add2(cnts[k], m);
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        float l0, l1, n0, n1;
        unpair(log2s[k], l0, l1);
        unpair(cnts[k], n0, n1);
        s_log[k] = l0 + l1;
        cnt[k] = n0 + n1;
    }
}
// Tail sums for any threshold, of log2(|g| * inv) with inv about 1 / g_min.  A NaN is not in the tail; an Inf makes s_log infinite.
template <bool BF16>
__device__ __forceinline__ void tail_any(const Words& w, float g_min, float inv, float& s_log, uint32_t& cnt) {
    float s[2] = {0.0f, 0.0f};
    cnt = 0;
    constexpr int n = kChunk<BF16>;
#pragma unroll
    for (int i = 0; i < n; ++i) {
        const uint32_t v = w[BF16 ? i / 2 : i];
        const float a = BF16 ? __uint_as_float((i & 1) ? (v & 0xFFFF0000u) : (v << 16)) : fabsf(__uint_as_float(v));
        const bool in_tail = a > g_min;
        const float lg = lg2_fast(a * inv);
        s[BF16 ? i & 1 : 0] += in_tail ? lg : 0.0f;          // at most 16 terms in a row
        cnt += in_tail ? 1u : 0u;
    }
    s_log = s[0] + s[1];
}

// Elements one by one in fp64: chunks with something non-finite, and a row's last d % chunk elements.  Out of line: the double-precision logarithm is long and needed rarely.
struct Exact {
    double sum_abs, sum_sq, sum_log2;
    uint32_t n_tail, n_bad;
    float max_abs;
};
template <bool BF16>
__device__ __noinline__ Exact exact_sums(const char* row, uint64_t first, uint32_t count, float t, float inv) {
    Exact r{0.0, 0.0, 0.0, 0u, 0u, 0.0f};
    for (uint32_t i = 0; i < count; ++i) {
        const float a = fabsf(load1<BF16>(row, first + i));
        if (!(a <= kMaxFinite)) { r.n_bad += 1; continue; }
        r.sum_abs += a;
        r.sum_sq += static_cast<double>(a) * a;
        r.max_abs = fmaxf(r.max_abs, a);
        if (a > t) { r.sum_log2 += log2(static_cast<double>(a) * static_cast<double>(inv)); r.n_tail += 1; }
    }
    return r;
}

// ---- what a thread has gathered, and its reduction over the block ------------------------------------------
template <bool BF16>
struct Gathered {
    double sum_abs = 0.0, sum_sq = 0.0, sum_log2[2] = {0.0, 0.0};
    float n_tail[2] = {0.0f, 0.0f};            // whole numbers below 2^24: a thread sees at most 2^40 / (2 * 148 * 256) elements
    unsigned long long n_bad = 0;
    uint32_t max_bits = 0;

    __device__ __forceinline__ void take_exact(const Exact& e, bool with_moments, int k, bool with_tail) {
        if (with_moments) {
            sum_abs += e.sum_abs; sum_sq += e.sum_sq; n_bad += e.n_bad;
            if constexpr (BF16) max_bits = max_b2(max_bits, __float_as_uint(e.max_abs) >> 16);
            else max_bits = __float_as_uint(fmaxf(__uint_as_float(max_bits), e.max_abs));
        }
        if (with_tail) { sum_log2[k] += e.sum_log2; n_tail[k] += static_cast<float>(e.n_tail); }
    }
    __device__ __forceinline__ Partial partial() const {
        Partial p;
        p.sum_abs = sum_abs; p.sum_sq = sum_sq; p.sum_log2[0] = sum_log2[0]; p.sum_log2[1] = sum_log2[1];
        p.n_tail[0] = static_cast<unsigned long long>(n_tail[0]); p.n_tail[1] = static_cast<unsigned long long>(n_tail[1]);
        p.n_bad = n_bad; p.max_abs = max_value<BF16>(max_bits); p.pad = 0.0f;
        return p;
    }
};
template <int WARPS>
struct BlockFold {
    double d[4][WARPS];
    unsigned long long u[3][WARPS];
    float f[WARPS];
    Partial total;
    bool last;
};
// Every thread passes its values; thread 0 gets the block's.  MOMENTS / TAILS say which fields are in use (TAILS: how many
// thresholds).  One block barrier; the shared arrays may be reused after the next one.  FEW: a thread's counts are what it
// has seen itself, below 2^24, so a warp's fit 32 bits (the bf16 hinted kernel does without: its main loop then gets other
// registers and takes 410 us instead of 404 on 124 M x 8).  The warps' values are added by the lanes of the first: with one thread
// taking them in turn two passes over 1 M x 8 took 0.4 us more, over 3.5 M bf16 x 1 0.3 us.
template <int WARPS, bool MOMENTS, int TAILS, bool FEW = true>
__device__ __forceinline__ void block_fold(Partial& p, BlockFold<WARPS>& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto count = [](unsigned long long v) -> unsigned long long {
        if constexpr (FEW) return __reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(v));
        else return warp_sum(v);
    };
    if constexpr (MOMENTS) {
        p.sum_abs = warp_sum(p.sum_abs); p.sum_sq = warp_sum(p.sum_sq); p.n_bad = count(p.n_bad); p.max_abs = warp_max_abs(p.max_abs);
    }
#pragma unroll
    for (int k = 0; k < TAILS; ++k) { p.sum_log2[k] = warp_sum(p.sum_log2[k]); p.n_tail[k] = count(p.n_tail[k]); }
    if (lane == 0) {
        if constexpr (MOMENTS) { sh.d[0][warp] = p.sum_abs; sh.d[1][warp] = p.sum_sq; sh.u[2][warp] = p.n_bad; sh.f[warp] = p.max_abs; }
#pragma unroll
        for (int k = 0; k < TAILS; ++k) { sh.d[2 + k][warp] = p.sum_log2[k]; sh.u[k][warp] = p.n_tail[k]; }
    }
    __syncthreads();
    if (warp == 0) {                                           // lane w: warp w's values
        Partial r{};
        if (lane < WARPS) {
            if constexpr (MOMENTS) { r.sum_abs = sh.d[0][lane]; r.sum_sq = sh.d[1][lane]; r.n_bad = sh.u[2][lane]; r.max_abs = sh.f[lane]; }
#pragma unroll
            for (int k = 0; k < TAILS; ++k) { r.sum_log2[k] = sh.d[2 + k][lane]; r.n_tail[k] = sh.u[k][lane]; }
        }
        if constexpr (MOMENTS) {
            r.sum_abs = warp_sum<WARPS>(r.sum_abs); r.sum_sq = warp_sum<WARPS>(r.sum_sq); r.n_bad = warp_sum<WARPS>(r.n_bad);
            r.max_abs = warp_max_abs(r.max_abs);
        }
#pragma unroll
        for (int k = 0; k < TAILS; ++k) { r.sum_log2[k] = warp_sum<WARPS>(r.sum_log2[k]); r.n_tail[k] = warp_sum<WARPS>(r.n_tail[k]); }
        if (lane == 0) p = r;
    }
}
constexpr int kWarps = kThreads / 32;

// Largest power of two not above x; 0 below the smallest normal number (no tail), Inf for Inf.
__device__ __forceinline__ float pow2_floor(float x) {
    return x >= 1.17549435e-38f ? __uint_as_float(__float_as_uint(x) & 0xFF800000u) : 0.0f;
}
__device__ __forceinline__ float mean_level(float kappa, double sum_abs, uint64_t d) {
    return d ? static_cast<float>(static_cast<double>(kappa) * sum_abs / static_cast<double>(d)) : 0.0f;
}
// Tail elements are scaled by inv before the logarithm and the exact logarithm of inv * g_min is taken out again at
// the end, so inv only has to keep |g| * inv inside the normal range for |g| > g_min.  1 / g_min overflows for a
// subnormal g_min; such a threshold is scaled by 2^64 first.
__device__ __forceinline__ float inverse_of(float g_min) {
    return g_min > 0.0f ? __frcp_rn(g_min < 7.8886090522101181e-31f ? g_min * 18446744073709551616.0f : g_min) : 0.0f;
}
__device__ __forceinline__ void store_moments(tq_stats_t* st, uint64_t d, const Partial& t, float g_min) {
    st->d = d; st->n_nonfinite = t.n_bad; st->sum_abs = t.sum_abs; st->sum_sq = t.sum_sq; st->max_abs = t.max_abs;
    st->g_min = g_min; st->reserved = 0;
}
// sum_log2 holds the logarithms of |g| * inv
__device__ __forceinline__ void store_tail(tq_stats_t* st, unsigned long long n, double sum_log2, float g_min, float inv) {
    const double corr = n ? static_cast<double>(n) * log2(static_cast<double>(inv) * static_cast<double>(g_min)) : 0.0;
    st->n_tail = n;
    st->sum_log_tail = (sum_log2 - corr) * 0.6931471805599453094;
}
// sum_log2 holds the logarithms of |g|, g_min is a power of two: log2 g_min is an integer
__device__ __forceinline__ void store_tail_pow2(tq_stats_t* st, unsigned long long n, double sum_log2, float g_min) {
    const int e2 = static_cast<int>((__float_as_uint(g_min) >> 23) & 0xFFu) - 127;
    st->n_tail = n;
    st->sum_log_tail = n ? (sum_log2 - static_cast<double>(n) * static_cast<double>(e2)) * 0.6931471805599453094 : 0.0;
}

// ---- a thread's share of a set of chunks ---------------------------------------------------------------------
enum Pass { kMoments = 0, kTail = 1, kBoth = 2 };

// Threshold g_min (any value; no tail unless positive).
template <bool BF16, int PASS>
__device__ __forceinline__ void take_any(const char* row, uint64_t c, Words& w, float g_min, float inv, Gathered<BF16>& g) {
    drop_signs<BF16>(w);
    float s_abs = 0.0f, s_sq = 0.0f, s_log = 0.0f;
    uint32_t cnt = 0;
    if constexpr (PASS != kTail) moments<BF16>(w, s_abs, s_sq);
    if constexpr (PASS != kMoments) {
        if (g_min > 0.0f) tail_any<BF16>(w, g_min, inv, s_log, cnt);
    }
    if ((s_abs + s_sq) <= kMaxFinite && fabsf(s_log) <= kMaxFinite) {
        if constexpr (PASS != kTail) { g.sum_abs += s_abs; g.sum_sq += s_sq; g.max_bits = chunk_max<BF16>(w, g.max_bits); }
        if constexpr (PASS != kMoments) { g.sum_log2[0] += s_log; g.n_tail[0] += static_cast<float>(cnt); }
    } else {
        g.take_exact(exact_sums<BF16>(row, c * kChunk<BF16>, kChunk<BF16>, PASS != kMoments && g_min > 0.0f ? g_min : CUDART_INF_F, inv),
                     PASS != kTail, 0, PASS != kMoments);
    }
}
// K thresholds t, 2 t that are powers of two (t = Inf: none), with the moments or without.
template <bool BF16, int K, bool MOMENTS>
__device__ __forceinline__ void take_pow2(const char* row, uint64_t c, Words& w, float t, const TailTest& test, Gathered<BF16>& g) {
    drop_signs<BF16>(w);
    float s_abs, s_sq, s_log[K], cnt[K];
    moments<BF16>(w, s_abs, s_sq);               // always: both forms send the same chunks through the exact path
    tail_pow2<BF16, K>(w, test, s_log, cnt);
    if ((s_abs + s_sq) <= kMaxFinite) {
        if constexpr (MOMENTS) { g.sum_abs += s_abs; g.sum_sq += s_sq; g.max_bits = chunk_max<BF16>(w, g.max_bits); }
#pragma unroll
        for (int k = 0; k < K; ++k) { g.sum_log2[k] += s_log[k]; g.n_tail[k] += cnt[k]; }
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k)
            g.take_exact(exact_sums<BF16>(row, c * kChunk<BF16>, kChunk<BF16>, k ? 2.0f * t : t, 1.0f), MOMENTS && k == 0, k, true);
    }
}
// A thread's chunks c, c + stride, ... below `end`.  One chunk at a time: with the loads of two issued together the registers
// cost a resident block, and the larger bursts made HBM slower (25.6 M x 16 fp32, two passes: 510 us instead of 481).
template <class Take>
__device__ __forceinline__ void walk(const char* row, uint64_t c, uint64_t end, uint32_t stride, const Take& take) {
    for (; c < end; c += stride) {
        Words w;
        load_chunk(row, c, w);
        take(c, w);
    }
}
template <bool BF16>
__device__ __forceinline__ uint64_t chunk_end_of(const JobPiece& piece) {
    const uint64_t whole = piece.d / kChunk<BF16>, end = piece.tile1 * kThreads;
    return end < whole ? end : whole;
}
// The row's last d % chunk elements, one for each of the first threads.
template <bool BF16>
__device__ __forceinline__ bool has_leftover(uint64_t d, uint64_t& j) {
    j = d / kChunk<BF16> * kChunk<BF16> + threadIdx.x;
    return j < d;
}
// ---- how the work is cut ------------------------------------------------------------------------------------
// Ranges (TilePlan), or blocks that keep to one job each: see plan_stats.
struct StatsPlan : TilePlan {
    uint32_t per_row;                              // blocks per worker where every block has one piece; 0: ranges
    uint32_t block_begin[TQ_MAX_SEGMENTS + 1];     // then: first block of each segment within the worker's blocks
};
__device__ __forceinline__ void range_of_block(const TilePlan& plan, uint32_t b, uint64_t& cur, uint64_t& end) {
    cur = first_tile_of_block(plan, b);
    end = first_tile_of_block(plan, b + 1);
}
__device__ __forceinline__ void range_of_block(const StatsPlan& plan, uint32_t b, uint64_t& cur, uint64_t& end) {
    if (plan.per_row == 0) return range_of_block(static_cast<const TilePlan&>(plan), b, cur, end);
    const uint32_t worker = b / plan.per_row, in_row = b - worker * plan.per_row;
    uint32_t seg = 0;
    while (seg + 8 < plan.segs.n && plan.block_begin[seg + 8] <= in_row) seg += 8;
    while (seg + 1 < plan.segs.n && plan.block_begin[seg + 1] <= in_row) ++seg;
    const uint32_t parts = plan.block_begin[seg + 1] - plan.block_begin[seg], part = in_row - plan.block_begin[seg];
    const uint64_t first = worker * plan.per_worker + plan.begin[seg], tiles = plan.begin[seg + 1] - plan.begin[seg];
    cur = first + tiles * part / parts;
    end = first + tiles * (part + 1) / parts;
}

template <bool BF16>
__device__ __forceinline__ const char* row_of(const JobPiece& piece, const void* grad, uint64_t grad_stride) {
    return static_cast<const char*>(grad) + (static_cast<uint64_t>(piece.worker) * grad_stride + piece.off) * (BF16 ? 2 : 4);
}
__device__ __forceinline__ Partial* records_of_job(const TilePlan& plan, const JobPiece& piece, Partial* partials, uint32_t& count) {
    uint32_t first, last;
    blocks_of_job(plan, piece, first, last);
    count = last - first + 1;
    return partials + first + piece.job;
}
__device__ __forceinline__ Partial* records_of_job(const StatsPlan& plan, const JobPiece& piece, Partial* partials, uint32_t& count) {
    if (plan.per_row == 0) return records_of_job(static_cast<const TilePlan&>(plan), piece, partials, count);
    count = plan.block_begin[piece.seg + 1] - plan.block_begin[piece.seg];
    return partials + piece.worker * plan.per_row + plan.block_begin[piece.seg] + piece.job;
}
__device__ __forceinline__ Partial* record_of_piece(const JobPiece& piece, Partial* partials) { return partials + blockIdx.x + piece.job; }
// Folds `count` records of an earlier launch (or of blocks whose tickets have been seen).
template <bool MOMENTS, int TAILS>
__device__ __forceinline__ void fold_records(const Partial* records, uint32_t count, Partial& p, BlockFold<kWarps>& sh) {
    p = Partial{};
    for (uint32_t b = threadIdx.x; b < count; b += kThreads) {
        const volatile Partial* q = records + b;
        if constexpr (MOMENTS) { p.sum_abs += q->sum_abs; p.sum_sq += q->sum_sq; p.n_bad += q->n_bad; p.max_abs = fmaxf(p.max_abs, q->max_abs); }
#pragma unroll
        for (int k = 0; k < TAILS; ++k) { p.sum_log2[k] += q->sum_log2[k]; p.n_tail[k] += q->n_tail[k]; }
    }
    block_fold<kWarps, MOMENTS, TAILS, false>(p, sh);
}
// The sum of |g| over the records, known to every thread; added as fold_records adds it, because a threshold that follows from the
// one has to equal that from the other.
__device__ __forceinline__ double fold_sum_abs(const Partial* records, uint32_t count, BlockFold<kWarps>& sh) {
    const int lane = threadIdx.x & 31;
    double v = 0.0;
    for (uint32_t b = threadIdx.x; b < count; b += kThreads) v += records[b].sum_abs;
    v = warp_sum(v);
    if (lane == 0) sh.d[0][threadIdx.x >> 5] = v;
    __syncthreads();
    static_assert(kWarps == 8, "");
    const double* d = sh.d[0];                                 // the tree of block_fold, without its shuffles
    v = ((d[0] + d[4]) + (d[2] + d[6])) + ((d[1] + d[5]) + (d[3] + d[7]));
    __syncthreads();
    return v;
}
// Stores the tail fields of the block's record and says whether all of the job's have been stored (block-uniform).
__device__ __forceinline__ bool last_of_job(Partial* record, const Partial& p, uint32_t* ticket, uint32_t count, BlockFold<kWarps>& sh) {
    if (threadIdx.x == 0) {
        record->sum_log2[0] = p.sum_log2[0]; record->n_tail[0] = p.n_tail[0];
        __threadfence();                                       // record visible before the ticket
        sh.last = atomicAdd(ticket, 1u) == count - 1;
    }
    __syncthreads();
    if (sh.last) __threadfence();
    return sh.last;
}

// ---- any threshold: moments, then tail; or both at once with the caller's ------------------------------------

// Resident blocks per SM, each with one range.  Measured with 3 / 4 / 5 blocks: 25.6 M x 16 fp32, two passes 482 / 477 / 506 us,
// hinted 258 / 247 / 273 (HBM: 250 us a pass); 124 M x 8 bf16, two passes 668 / 623 / 622 us, hinted 456 / 430 / 470 (555 before; the
// special-function unit, one log2 per element, is busy 54 % of the time, the multiply-add pipes 57 %, issue 69 %).
constexpr int kStatsBlocksPerSm = 4;

template <bool BF16, int PASS>
__device__ __forceinline__ void stats_piece(const JobPiece& piece, const StatsPlan& plan, const void* grad, uint64_t grad_stride, float g_min,
                                            float kappa, tq_stats_t* stats, Partial* partials, uint32_t* tickets, BlockFold<kWarps>& sh) {
    const char* row = row_of<BF16>(piece, grad, grad_stride);
    uint32_t count;
    const Partial* records = records_of_job(plan, piece, partials, count);
    if constexpr (PASS == kMoments) {
        if (piece.tile0 == 0 && threadIdx.x == 0) tickets[piece.job] = 0u;          // for the tail pass
    }
    if constexpr (PASS == kTail) {
        // finish the moments: every piece needs the threshold, the job's first one writes the record
        if (piece.tile0 == 0) {
            Partial t;
            fold_records<true, 0>(records, count, t, sh);
            if (threadIdx.x == 0) {
                sh.total = t;
                store_moments(stats + piece.job, piece.d, t, mean_level(kappa, t.sum_abs, piece.d));
            }
            __syncthreads();
            g_min = mean_level(kappa, sh.total.sum_abs, piece.d);
        } else {
            g_min = mean_level(kappa, fold_sum_abs(records, count, sh), piece.d);
        }
    }
    const float inv = PASS == kMoments ? 0.0f : inverse_of(g_min);
    Gathered<BF16> g;
    walk(row, piece.tile0 * kThreads + threadIdx.x, chunk_end_of<BF16>(piece), kThreads,
         [&](uint64_t c, Words& w) { take_any<BF16, PASS>(row, c, w, g_min, inv, g); });
    uint64_t j;
    if (piece.last && has_leftover<BF16>(piece.d, j))
        g.take_exact(exact_sums<BF16>(row, j, 1, PASS != kMoments && g_min > 0.0f ? g_min : CUDART_INF_F, inv), PASS != kTail, 0, PASS != kMoments);

    Partial p = g.partial();
    block_fold<kWarps, PASS != kTail, PASS != kMoments ? 1 : 0>(p, sh);
    if constexpr (PASS != kTail) {
        if (threadIdx.x == 0) *record_of_piece(piece, partials) = p;
    } else {
        if (!last_of_job(record_of_piece(piece, partials), p, tickets + piece.job, count, sh)) return;
        Partial t;
        fold_records<false, 1>(records, count, t, sh);
        if (threadIdx.x == 0) store_tail(stats + piece.job, t.n_tail[0], t.sum_log2[0], g_min, inv);
    }
}

template <bool BF16, int PASS>
__global__ void __launch_bounds__(kThreads, kStatsBlocksPerSm)
stats_kernel(const void* __restrict__ grad, uint64_t grad_stride, float g_min, float kappa, tq_stats_t* stats, Partial* partials,
             uint32_t* tickets, const __grid_constant__ StatsPlan plan) {
    __shared__ BlockFold<kWarps> sh;
    uint64_t cur, end;
    range_of_block(plan, blockIdx.x, cur, end);
    JobPiece piece = next_piece(plan, cur, end);               // no block is empty
    pdl_wait();
    while (true) {
        stats_piece<BF16, PASS>(piece, plan, grad, grad_stride, g_min, kappa, stats, partials, tickets, sh);
        if (cur >= end) break;
        __syncthreads();                                       // the next piece reuses the shared arrays
        piece = next_piece(plan, cur, end);
    }
}

// The records of a pass with the caller's threshold, a block per job.  As tickets of that pass, with the last block of a job folding,
// each piece of a block waited for the one before it, and the first for a memset (8 rows of 1 M in 16 groups 20.5 us, now 10.9; 25.6 M x 16
// 242, now 239).
__global__ void __launch_bounds__(kThreads)
stats_given_finish_kernel(float g_min, tq_stats_t* stats, Partial* partials, const __grid_constant__ StatsPlan plan) {
    __shared__ BlockFold<kWarps> sh;
    const uint32_t worker = blockIdx.x / plan.segs.n, seg = blockIdx.x - worker * plan.segs.n;
    uint64_t cur = worker * plan.per_worker + plan.begin[seg];
    const JobPiece job = next_piece(plan, cur, cur + 1);
    uint32_t count;
    const Partial* records = records_of_job(plan, job, partials, count);
    pdl_wait();
    Partial t;
    fold_records<true, 1>(records, count, t, sh);
    if (threadIdx.x == 0) {
        store_moments(stats + job.job, job.d, t, g_min);
        store_tail(stats + job.job, t.n_tail[0], t.sum_log2[0], g_min, inverse_of(g_min));
    }
}

// ---- hinted threshold -----------------------------------------------------------------------------------------
// The paper leaves the choice of g_min open (Section 4.1 only calls it the lower end of the power-law range); with g_min =
// kappa * mean|g| rounded DOWN TO A POWER OF TWO the tail sums can be gathered before the mean is known, for two
// candidate powers of two at once: a caller-kept hint (the kappa * mean|g| of the previous round) names the two
// candidates nearest to it, and the launch that folds the records keeps the candidate that the finished mean selects.
// If neither fits (first round, or the mean moved by more than a factor of about 1.4 to 2), that launch redoes the tail sums for the
// right threshold, so the host never has to look.  The sums of one threshold are the same, bit for bit, whichever way
// they were obtained: both sum log2|g| itself and take n * log2(g_min), an integer multiple, out at the end.

// Smaller candidate for a hint; the other one is twice that.  Inf: no hint.
__device__ __forceinline__ float lower_candidate(float level) {
    if (!(level >= 2.3509887e-38f && level <= kMaxFinite)) return CUDART_INF_F;      // from 2^-125: both candidates are normal numbers
    const uint32_t bits = __float_as_uint(level), e = bits & 0x7F800000u;
    return __uint_as_float((bits & 0x00400000u) ? e : e - 0x00800000u);             // mantissa >= 1.5: {2^h, 2^(h+1)}, else {2^(h-1), 2^h}
}
// Which of the candidates t, 2 t is the threshold: 0, 1, -1 neither, 2 there is no tail at all.
__device__ __forceinline__ int candidate_of(float g_min, float t) {
    return !(g_min > 0.0f && g_min <= kMaxFinite) ? 2 : g_min == t ? 0 : g_min == 2.0f * t ? 1 : -1;
}

template <bool BF16>
__device__ __forceinline__ void hinted_piece(const JobPiece& piece, const void* grad, uint64_t grad_stride,
                                             const tq_gmin_hint_t* hint, Partial* partials, uint32_t* tickets, BlockFold<kWarps>& sh) {
    const char* row = row_of<BF16>(piece, grad, grad_stride);
    const float t = lower_candidate(hint[piece.job].level);
    const TailTest test(t);
    Gathered<BF16> g;
    walk(row, piece.tile0 * kThreads + threadIdx.x, chunk_end_of<BF16>(piece), kThreads,
         [&](uint64_t c, Words& w) { take_pow2<BF16, 2, true>(row, c, w, t, test, g); });
    uint64_t j;
    if (piece.last && has_leftover<BF16>(piece.d, j)) {
        g.take_exact(exact_sums<BF16>(row, j, 1, t, 1.0f), true, 0, true);
        g.take_exact(exact_sums<BF16>(row, j, 1, 2.0f * t, 1.0f), false, 1, true);
    }
    Partial p = g.partial();
    block_fold<kWarps, true, 2, !BF16>(p, sh);
    if (threadIdx.x == 0) {
        p.pad = hint[piece.job].level;                           // the finishing launch overwrites the hint
        *record_of_piece(piece, partials) = p;
        if (piece.tile0 == 0) tickets[piece.job] = 0u;           // for the finishing launch
    }
}

// What one warp makes of a job's records: the sum of |g|, and with ALL every other field too.  Same order in every warp.  Several records per lane
// are asked for before the first is added: one after the other, each a trip to the L2, the 428 records of one row of 3.5 M bf16 values took
// 4 us.
__device__ __forceinline__ void load_pair(const void* p, double& a, double& b) {      // past the L1: other blocks may have written since
    asm volatile("ld.volatile.global.v2.f64 {%0,%1}, [%2];" : "=d"(a), "=d"(b) : "l"(p));
}
template <bool ALL>
__device__ __forceinline__ Partial warp_fold(const Partial* records, uint32_t count) {
    const uint32_t lane = threadIdx.x & 31u;
    constexpr uint32_t kAhead = ALL ? 3 : 16;
    Partial p{};
    for (uint32_t first = lane; first < count; first += 32 * kAhead) {
        double v[kAhead][ALL ? 8 : 2];
#pragma unroll
        for (uint32_t i = 0; i < kAhead; ++i) {
            const uint32_t b = first + 32 * i;
#pragma unroll
            for (int f = 0; f < (ALL ? 8 : 2); f += 2) {
                v[i][f] = v[i][f + 1] = 0.0;
                if (b < count) load_pair(reinterpret_cast<const double*>(records + b) + f, v[i][f], v[i][f + 1]);
            }
        }
#pragma unroll
        for (uint32_t i = 0; i < kAhead; ++i) {
            p.sum_abs += v[i][0];
            if constexpr (ALL) {
                p.sum_sq += v[i][1]; p.sum_log2[0] += v[i][2]; p.sum_log2[1] += v[i][3];
                p.n_tail[0] += static_cast<unsigned long long>(__double_as_longlong(v[i][4]));
                p.n_tail[1] += static_cast<unsigned long long>(__double_as_longlong(v[i][5]));
                p.n_bad += static_cast<unsigned long long>(__double_as_longlong(v[i][6]));
                p.max_abs = fmaxf(p.max_abs, __int_as_float(__double2loint(v[i][7])));
            }
        }
    }
    p.sum_abs = __shfl_sync(0xFFFFFFFFu, warp_sum(p.sum_abs), 0);
    if constexpr (ALL) {
        p.sum_sq = warp_sum(p.sum_sq); p.n_bad = warp_sum(p.n_bad); p.max_abs = warp_max_abs(p.max_abs);
#pragma unroll
        for (int k = 0; k < 2; ++k) { p.sum_log2[k] = warp_sum(p.sum_log2[k]); p.n_tail[k] = warp_sum(p.n_tail[k]); }
    }
    return p;
}
// Finishes a piece as far as the first launch allows: by one warp, a block's pieces side by side.  The job's first piece writes the
// record.  Returns the threshold if the piece's tail has to be read again, else 0.
__device__ __forceinline__ float hinted_finish_piece(const JobPiece& piece, float kappa, tq_gmin_hint_t* hint_out,
                                                     tq_stats_t* stats, Partial* partials, const Partial* records, uint32_t count) {
    const float t = lower_candidate(record_of_piece(piece, partials)->pad);
    const bool first = piece.tile0 == 0;
    // a miss lets other blocks overwrite the tail fields of their records, which are then not used here
    const Partial r = first ? warp_fold<true>(records, count) : warp_fold<false>(records, count);
    const float level = mean_level(kappa, r.sum_abs, piece.d), g_min = pow2_floor(level);
    const int pick = candidate_of(g_min, t);
    if (first && (threadIdx.x & 31u) == 0) {
        tq_stats_t* st = stats + piece.job;
        store_moments(st, piece.d, r, g_min);
        hint_out[piece.job].level = level;
        hint_out[piece.job].hit = pick >= 0 ? 1u : 0u;
        if (pick == 2) store_tail_pow2(st, 0, 0.0, g_min);
        else if (pick >= 0) store_tail_pow2(st, pick ? r.n_tail[1] : r.n_tail[0], pick ? r.sum_log2[1] : r.sum_log2[0], g_min);
    }
    return pick >= 0 ? 0.0f : g_min;
}
// The tail sums of a piece of a job whose hint missed.
template <bool BF16>
__device__ __forceinline__ void hinted_tail_piece(const JobPiece& piece, const TilePlan& plan, const void* grad, uint64_t grad_stride, float g_min,
                                                  tq_stats_t* stats, Partial* partials, uint32_t* tickets, BlockFold<kWarps>& sh) {
    uint32_t count;
    const Partial* records = records_of_job(plan, piece, partials, count);
    const char* row = row_of<BF16>(piece, grad, grad_stride);
    const TailTest test(g_min);
    Gathered<BF16> g;
    walk(row, piece.tile0 * kThreads + threadIdx.x, chunk_end_of<BF16>(piece), kThreads,
         [&](uint64_t c, Words& w) { take_pow2<BF16, 1, false>(row, c, w, g_min, test, g); });
    uint64_t j;
    if (piece.last && has_leftover<BF16>(piece.d, j)) g.take_exact(exact_sums<BF16>(row, j, 1, g_min, 1.0f), false, 0, true);
    Partial p = g.partial();
    block_fold<kWarps, false, 1>(p, sh);
    if (!last_of_job(record_of_piece(piece, partials), p, tickets + piece.job, count, sh)) return;
    if (threadIdx.x < 32) {                                    // as hinted_finish_piece folds them, or the sums could differ in the last bit
        const Partial t = warp_fold<true>(records, count);
        if (threadIdx.x == 0) store_tail_pow2(stats + piece.job, t.n_tail[0], t.sum_log2[0], g_min);
    }
}

template <bool BF16>
__global__ void __launch_bounds__(kThreads, kStatsBlocksPerSm)
stats_hinted_kernel(const void* __restrict__ grad, uint64_t grad_stride, const tq_gmin_hint_t* hint, Partial* partials, uint32_t* tickets,
                    const __grid_constant__ TilePlan plan) {
    __shared__ BlockFold<kWarps> sh;
    pdl_wait();
    uint64_t cur, end;
    range_of_block(plan, blockIdx.x, cur, end);
    while (cur < end) {
        hinted_piece<BF16>(next_piece(plan, cur, end), grad, grad_stride, hint, partials, tickets, sh);
        __syncthreads();                                       // the next piece reuses the shared arrays
    }
}
template <bool BF16>
__global__ void __launch_bounds__(kThreads, kStatsBlocksPerSm)
stats_hinted_finish_kernel(const void* __restrict__ grad, uint64_t grad_stride, float kappa, tq_gmin_hint_t* hint, tq_stats_t* stats,
                           Partial* partials, uint32_t* tickets, const __grid_constant__ TilePlan plan) {
    __shared__ BlockFold<kWarps> sh;
    __shared__ float s_again[kWarps];
    const uint32_t warp = threadIdx.x >> 5;
    uint64_t cur, end, batch;
    range_of_block(plan, blockIdx.x, cur, end);
    JobPiece mine;
    const Partial* records = nullptr;
    uint32_t n, count = 0;
    auto next_batch = [&] {                                    // as many pieces at a time as the block has warps
        batch = cur;
        for (n = 0; cur < end && n < kWarps; ++n) {
            const JobPiece piece = next_piece(plan, cur, end);
            if (n == warp) { mine = piece; records = records_of_job(plan, mine, partials, count); }
        }
    };
    next_batch();                                              // which are known before the records are there
    pdl_wait();
    while (true) {
        if (warp < n) {
            const float again = hinted_finish_piece(mine, kappa, hint, stats, partials, records, count);
            if ((threadIdx.x & 31u) == 0) s_again[warp] = again;
        }
        __syncthreads();
        uint64_t redo = batch;
        for (uint32_t i = 0; i < n; ++i) {
            const JobPiece piece = next_piece(plan, redo, end);
            if (s_again[i] > 0.0f) {
                hinted_tail_piece<BF16>(piece, plan, grad, grad_stride, s_again[i], stats, partials, tickets, sh);
                __syncthreads();
            }
        }
        if (cur >= end) break;
        __syncthreads();
        next_batch();
    }
}

// ---- short rows: one cluster per job, one launch -----------------------------------------------------------------
constexpr int kCluster = 8, kSmallThreads = 512, kSmallWarps = kSmallThreads / 32;
constexpr int kSmallChunks = 4;              // most per thread

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <class T>
__device__ __forceinline__ T of_rank(const T& mine, uint32_t rank) {          // the same shared variable of another block of the cluster
    static_assert(sizeof(T) == 4 || sizeof(T) == 8, "");
    uint32_t addr;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(addr) : "r"(smem_addr(&mine)), "r"(rank));
    if constexpr (sizeof(T) == 8) {
        unsigned long long v;
        asm volatile("ld.shared::cluster.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
        return __builtin_bit_cast(T, v);
    } else {
        uint32_t v;
        asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
        return __builtin_bit_cast(T, v);
    }
}

// A thread's CHUNKS chunks stay in registers between the two passes (one kernel for 4 chunks is 0.3 us slower on rows of
// up to 2, reading the third and fourth again 0.7 us on the others).
enum Rule { kGiven, kMean, kPow2 };    // g_min: the caller's; kappa * mean|g|; that rounded down to a power of two (the hint is kept up, not needed)
template <bool BF16, int RULE, int CHUNKS>
__global__ void __cluster_dims__(kCluster, 1, 1) __launch_bounds__(kSmallThreads)
stats_small_kernel(const void* __restrict__ grad, uint64_t grad_stride, float g_min, float kappa, tq_gmin_hint_t* hint, tq_stats_t* stats,
                   const __grid_constant__ SegTable segs) {
    __shared__ BlockFold<kSmallWarps> sh;
    __shared__ Partial s_moments, s_tail;
    pdl_wait();
    const uint32_t job = blockIdx.x / kCluster, rank = blockIdx.x % kCluster, worker = job / segs.n, seg = job - worker * segs.n;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t d = segs.len[seg], n_chunks = d / kChunk<BF16>;
    const char* row = static_cast<const char*>(grad) + (static_cast<uint64_t>(worker) * grad_stride + segs.off[seg]) * (BF16 ? 2 : 4);
    constexpr uint32_t stride = kCluster * kSmallThreads;
    const uint64_t c0 = rank * kSmallThreads + threadIdx.x;
    Words w[CHUNKS];
#pragma unroll
    for (int i = 0; i < CHUNKS; ++i)
        if (c0 + i * stride < n_chunks) load_chunk(row, c0 + i * stride, w[i]);
    uint64_t j;
    const bool leftover = rank == kCluster - 1 && has_leftover<BF16>(d, j);

    Gathered<BF16> g;
#pragma unroll
    for (int i = 0; i < CHUNKS; ++i)
        if (c0 + i * stride < n_chunks) take_any<BF16, RULE == kGiven ? kBoth : kMoments>(row, c0 + i * stride, w[i], g_min, inverse_of(g_min), g);
    if (leftover) g.take_exact(exact_sums<BF16>(row, j, 1, RULE == kGiven ? g_min : CUDART_INF_F, inverse_of(g_min)), true, 0, RULE == kGiven);
    Partial p = g.partial();
    block_fold<kSmallWarps, true, RULE == kGiven ? 1 : 0>(p, sh);
    if (threadIdx.x == 0) { s_moments = p; if constexpr (RULE == kGiven) s_tail = p; }
    cluster_sync();

    auto over_ranks = [&](auto v) {                            // lanes 0..7 hold one block's value each
        v = lane < kCluster ? v : decltype(v)(0);
#pragma unroll
        for (int o = kCluster / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
        return __shfl_sync(0xFFFFFFFFu, v, 0);
    };
    const uint32_t from = lane % kCluster;
    const double sum_abs = over_ranks(of_rank(s_moments.sum_abs, from));      // every warp for itself, in the same order
    const float level = mean_level(kappa, sum_abs, d);
    if constexpr (RULE == kPow2) g_min = pow2_floor(level);
    if constexpr (RULE == kMean) g_min = level;
    const bool tail_on = g_min > 0.0f && g_min <= kMaxFinite;
    const float inv = inverse_of(g_min);
    const TailTest test(g_min);

    if constexpr (RULE != kGiven) {
        g = Gathered<BF16>();
        if (tail_on) {
#pragma unroll
            for (int i = 0; i < CHUNKS; ++i) {
                const uint64_t c = c0 + i * stride;
                if (c >= n_chunks) continue;
                if constexpr (RULE == kPow2) take_pow2<BF16, 1, false>(row, c, w[i], g_min, test, g);
                else take_any<BF16, kTail>(row, c, w[i], g_min, inv, g);
            }
            if (leftover) g.take_exact(exact_sums<BF16>(row, j, 1, g_min, RULE == kPow2 ? 1.0f : inv), false, 0, true);
        }
        p = g.partial();
        block_fold<kSmallWarps, false, 1>(p, sh);
        if (threadIdx.x == 0) s_tail = p;
        cluster_sync();
    }
    if (rank == 0 && threadIdx.x < 32) {
        Partial t{};
        t.sum_abs = sum_abs;
        t.sum_sq = over_ranks(of_rank(s_moments.sum_sq, from));
        t.n_bad = over_ranks(of_rank(s_moments.n_bad, from));
        t.max_abs = warp_max_abs(of_rank(s_moments.max_abs, from));
        const unsigned long long n = over_ranks(of_rank(s_tail.n_tail[0], from));
        const double sum_log2 = over_ranks(of_rank(s_tail.sum_log2[0], from));
        if (lane == 0) {
            store_moments(stats + job, d, t, g_min);
            if constexpr (RULE == kPow2) {
                store_tail_pow2(stats + job, n, sum_log2, g_min);
                hint[job].hit = candidate_of(g_min, lower_candidate(hint[job].level)) >= 0 ? 1u : 0u;      // as the long form reports it
                hint[job].level = level;
            } else {
                store_tail(stats + job, n, sum_log2, g_min, inv);
            }
        }
    }
    cluster_sync();                                            // no block leaves while another reads its shared memory
}

// ---- launches -----------------------------------------------------------------------------------------------------

// Rows of at most this many bytes, in calls whose clusters are resident at the same time, take the cluster kernel.  Device
// time against the two launches (hinted / two-pass): 100 k x 1 fp32 6.5 / 6.4 against 8.0 / 8.5 us, 250 k x 8 10.9 / 10.3 against
// 11.5 / 12.7; beyond, the few SMs of a cluster are too slow (500 k x 1: 13.2 against 9.0 us) or the clusters queue
// (250 k x 16: 18.7 against 13.9 us).  One launch less on the host (2.5 us) comes on top.
constexpr uint64_t kSmallRowBytes = static_cast<uint64_t>(kCluster) * kSmallThreads * kSmallChunks * kChunkBytes;      // 1 MiB
constexpr uint32_t kSmallMaxJobs = 8;

// Where layer groups are short, the pieces of a range stand in a chain: in the tail pass each folds its job's records and ends with a
// ticket.  Calls without a hint whose resident blocks would get up to 8 tiles give each block a piece of one job instead, of
// about 1.25 times an even share (fewer blocks than places where jobs allow it, so that one wave holds them).  Ranges / one job each,
// us: two passes over 32 rows of 500 k in 30 groups 56.1 / 30.1, 64 x 200 k in 40 60.2 / 45.7, 8 x 1 M in 40 30.1 / 18.4; threshold given
// 23.1 / 20.4, 30.9 / 27.4, 12.5 / 10.3.  From 14 tiles on ranges are faster (11 x 3 M fp32 in 16, threshold given: 27.4 / 31.9), as they are
// behind a hint, whose records a block folds side by side (64 x 200 k in 40: 32.2 / 36.0); its kernels do not
// know the other form, which moved the registers of the bf16 main loop (38 M x 11: 579 -> 587 us a round).
constexpr uint64_t kTilesForRanges = 8;

static uint64_t resident_blocks(uint32_t n_jobs) {
    const uint64_t resident = static_cast<uint64_t>(sm_count()) * kStatsBlocksPerSm, room = static_cast<uint64_t>(n_jobs) * kRecordsPerJob - n_jobs;
    return resident < room ? resident : room;
}
static void plan_ranges(const StatsCall& c, uint32_t n_jobs, TilePlan* plan) {
    const uint64_t resident = resident_blocks(n_jobs), room = static_cast<uint64_t>(n_jobs) * kRecordsPerJob - n_jobs;
    plan_tiles(plan, c.segs, c.d, c.n_workers, kThreads * kChunkBytes / (c.bf16 ? 2 : 4), resident);
    // bf16 rows are bound by instructions: three ranges per resident block even out the SMs (124 M x 8, hinted: 430 -> 407 us;
    // fp32 rows 249 -> 254 us, short ranges lose more)
    if (c.bf16 && plan->per_block >= 64 && 3 * resident <= room) plan_tiles(plan, c.segs, c.d, c.n_workers, kThreads * kChunkBytes / 2, 3 * resident);
}
static void plan_stats(const StatsCall& c, uint32_t n_jobs, StatsPlan* plan) {
    plan_ranges(c, n_jobs, plan);
    plan->per_row = 0;
    const uint64_t total = plan->per_worker * c.n_workers, resident = resident_blocks(n_jobs);
    if (plan->segs.n == 1 || total <= resident || total > kTilesForRanges * resident) return;
    const uint64_t target = total * 5 / (resident * 4);          // at least 1
    uint32_t blocks = 0;
    for (uint32_t s = 0; s < plan->segs.n; ++s) {
        plan->block_begin[s] = blocks;
        const uint64_t parts = (plan->begin[s + 1] - plan->begin[s] + target / 2) / target;
        blocks += parts > 0 ? static_cast<uint32_t>(parts) : 1u;
    }
    plan->block_begin[plan->segs.n] = plan->per_row = blocks;
    plan->blocks = blocks * c.n_workers;
}

// Equal rows in a whole number of blocks each may leave some places empty: see launch_kernel.  Rounds of 3 M x 64, 576 blocks of 81
// tiles, early / late: hinted 336 / 315 us, two passes 461 / 416; of 1 M x 64, 27 tiles, two passes 152.8 / 153.4.
static Start start_of(const TilePlan& plan) {
    return plan.blocks < static_cast<uint32_t>(sm_count()) * kStatsBlocksPerSm && plan.per_block >= 48 ? Start::kLate : Start::kEarly;
}

template <int RULE, int CHUNKS>
static cudaError_t launch_clusters(const StatsCall& c, uint32_t n_jobs, tq_gmin_hint_t* hint, const SegTable& segs) {
    return launch_kernel(c.bf16 ? stats_small_kernel<true, RULE, CHUNKS> : stats_small_kernel<false, RULE, CHUNKS>, dim3(n_jobs * kCluster), kSmallThreads,
                         0, c.stream, c.grad, c.grad_stride, c.g_min, c.kappa, hint, c.stats, segs);
}
// True when the call went to the cluster kernel.
template <int RULE>
static bool launch_small(const StatsCall& c, uint32_t n_jobs, tq_gmin_hint_t* hint, cudaError_t* e) {
    if (n_jobs > kSmallMaxJobs) return false;
    SegTable one;
    if (!c.segs) { one.n = 1; one.off[0] = 0; one.len[0] = c.d; }
    const SegTable& segs = c.segs ? *c.segs : one;
    uint64_t most = 0;
    for (uint32_t s = 0; s < segs.n; ++s) most = segs.len[s] > most ? segs.len[s] : most;
    most *= c.bf16 ? 2 : 4;
    if (most > kSmallRowBytes) return false;
    *e = most <= kSmallRowBytes / 2 ? launch_clusters<RULE, kSmallChunks / 2>(c, n_jobs, hint, segs) : launch_clusters<RULE, kSmallChunks>(c, n_jobs, hint, segs);
    return true;
}

cudaError_t launch_stats(const StatsCall& c, int* launches) {
    *launches = 0;
    const uint32_t n_jobs = c.segs ? c.n_workers * c.segs->n : c.n_workers;
    cudaError_t e;
    if (c.g_min > 0.0f ? launch_small<kGiven>(c, n_jobs, nullptr, &e) : launch_small<kMean>(c, n_jobs, nullptr, &e)) {
        *launches = e == cudaSuccess ? 1 : 0;
        return e;
    }
    Partial* partials = static_cast<Partial*>(c.workspace);
    uint32_t* tickets = reinterpret_cast<uint32_t*>(static_cast<char*>(c.workspace) + tickets_offset(n_jobs));
    static thread_local StatsPlan plan;
    plan_stats(c, n_jobs, &plan);
    auto launch = [&](auto kernel, Start start) {
        e = launch_kernel(start, kernel, dim3(plan.blocks), kThreads, 0, c.stream, c.grad, c.grad_stride, c.g_min, c.kappa, c.stats, partials, tickets, plan);
        *launches += e == cudaSuccess ? 1 : 0;
        return e;
    };
    if (c.g_min > 0.0f) {
        if (launch(c.bf16 ? stats_kernel<true, kBoth> : stats_kernel<false, kBoth>, start_of(plan)) != cudaSuccess) return e;
        e = launch_kernel(stats_given_finish_kernel, dim3(n_jobs), kThreads, 0, c.stream, c.g_min, c.stats, partials, plan);
        *launches += e == cudaSuccess ? 1 : 0;
        return e;
    }
    if (launch(c.bf16 ? stats_kernel<true, kMoments> : stats_kernel<false, kMoments>, start_of(plan)) != cudaSuccess) return e;
    return launch(c.bf16 ? stats_kernel<true, kTail> : stats_kernel<false, kTail>, Start::kEarly);
}

cudaError_t launch_stats_hinted(const StatsCall& c, tq_gmin_hint_t* hint, int* launches) {
    *launches = 0;
    const uint32_t n_jobs = c.segs ? c.n_workers * c.segs->n : c.n_workers;
    cudaError_t e;
    if (launch_small<kPow2>(c, n_jobs, hint, &e)) { *launches = e == cudaSuccess ? 1 : 0; return e; }
    Partial* partials = static_cast<Partial*>(c.workspace);
    uint32_t* tickets = reinterpret_cast<uint32_t*>(static_cast<char*>(c.workspace) + tickets_offset(n_jobs));
    static thread_local TilePlan plan;            // the same plan for both launches: same summation order
    plan_ranges(c, n_jobs, &plan);
    e = launch_kernel(start_of(plan), c.bf16 ? stats_hinted_kernel<true> : stats_hinted_kernel<false>, dim3(plan.blocks), kThreads, 0, c.stream, c.grad,
                      c.grad_stride, static_cast<const tq_gmin_hint_t*>(hint), partials, tickets, plan);
    if (e != cudaSuccess) return e;
    *launches = 1;
    e = launch_kernel(c.bf16 ? stats_hinted_finish_kernel<true> : stats_hinted_finish_kernel<false>, dim3(plan.blocks), kThreads, 0, c.stream,
                      c.grad, c.grad_stride, c.kappa, hint, c.stats, partials, tickets, plan);
    if (e == cudaSuccess) *launches = 2;
    return e;
}

// ---------------------------------------------------------------------------------------------
// Built-in scratch for callers that cannot allocate: enough for TQ_STATIC_MAX_WORKERS workers.
// It is part of the library's device image (one copy per GPU that loads the library).
constexpr size_t kStaticScratchBytes =
    static_cast<size_t>(TQ_STATIC_MAX_WORKERS) * kRecordsPerJob * sizeof(Partial) + TQ_STATIC_MAX_WORKERS * 2 * sizeof(uint32_t) + 256;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

cudaError_t launch_stats_static(const StatsCall& c, int* launches, bool* limit) {
    *launches = 0;
    *limit = c.n_workers > TQ_STATIC_MAX_WORKERS || stats_workspace_bytes(c.n_workers) > kStaticScratchBytes;
    if (*limit) return cudaSuccess;

    // In host code `g_static_scratch` is only a handle for the symbol, not a device address: the
    // address must be asked for, per device, with that device current.  Done on the first call
    // on each device and remembered.
    constexpr int kMaxDevices = 64;
    static void* s_addr[kMaxDevices] = {};
    static std::mutex s_lock;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    void* ptr = nullptr;
    {
        std::lock_guard<std::mutex> hold(s_lock);
        if (!s_addr[dev]) {
            e = cudaGetSymbolAddress(&ptr, g_static_scratch);
            if (e != cudaSuccess) return e;
            s_addr[dev] = ptr;
        }
        ptr = s_addr[dev];
    }
    StatsCall with_scratch = c;
    with_scratch.workspace = ptr;
    return launch_stats(with_scratch, launches);   // nothing in the scratch has to be cleared first
}

}  // namespace tq

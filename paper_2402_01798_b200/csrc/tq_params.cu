// Parameter design: statistics -> truncation threshold alpha and codebook, on the host (tq_params,
// tq_params_batch, tq_params_from_levels) and, with the same code, on the device (tq_params_device:
// one warp per worker, so a round needs no host round trip between statistics and compression).
//
// Follows Section 4 of the paper.  The gradient density is modelled as a power-law tail
// p(g) = rho (gamma-1) g_min^(gamma-1) |g|^-gamma beyond g_min (Section 4.1, tail model), with rho
// the one-sided tail mass, completed by a flat body p = (1 - 2 rho) / (2 g_min) below g_min so that
// Q_U, Q_N and the p^(1/3) density of Section 4.2 are defined on the whole of [-alpha, alpha].
// Everything here is O(L) double-precision work per worker; results are rounded once to fp32.
// Host and device use their own log / exp / cbrt, so the two can differ in the last fp32 bit
// of alpha or of a level; each is a valid quantizer, and a packed buffer is always decoded with the
// parameters it was encoded with.
//
// On the device this is one short chain of dependent double-precision functions, so its time is their
// latency times their number.  Hence: lengths are measured in units of g_min and by their logarithm
// x = ln(a / g_min), in which a boxed alpha equation costs one exp and one log; it is solved by Newton
// steps (4 to 8 evaluations); and everything that exists once per level or per trial point (levels, inverse
// widths, the split of the two-step quantizer) is spread over the lanes of the warp.  Measured on B200 for
// one worker, uniform, 4 levels / 8 workers, 16-level two-step quantizer: 4.5 us / 18.1 us, against
// 21.1 us / 3590 us with one thread per worker, two pow per evaluation and Aitken steps.  The two-step quantizer's
// trial points are the same for every alpha, so their powers k^-gamma are taken once (29.1 us with an exp
// and a division per point and alpha; on the host, where one thread does all of them, 22 -> 6.6 us per record).
#include <cmath>

#include "tq.h"
#include "tq_device.cuh"
#include "tq_launch.h"

namespace tq {

#define TQ_HD __host__ __device__

TQ_HD inline bool finite_f(float x) { return fabsf(x) <= 3.402823466e38f; }
TQ_HD inline bool finite_d(double x) { return fabs(x) <= 1.7976931348623157e308; }

// Who works on one record: the calling host thread alone, or the 32 lanes of a warp.  All lanes run the same
// scalar code; `ballot` collects one bit per lane (all lanes call it together).
struct OneThread {
    static constexpr int kLanes = 1;
    TQ_HD int lane() const { return 0; }
    TQ_HD uint32_t ballot(bool b) const { return b ? 1u : 0u; }
    TQ_HD double of(double v, int) const { return v; }          // another lane's value
    TQ_HD void sync() const {}
};
struct OneWarp {
    static constexpr int kLanes = 32;
#ifdef __CUDA_ARCH__
    __device__ int lane() const { return static_cast<int>(threadIdx.x & 31u); }
    __device__ uint32_t ballot(bool b) const { return __ballot_sync(0xFFFFFFFFu, b); }
    __device__ double of(double v, int lane) const { return __shfl_sync(0xFFFFFFFFu, v, lane); }
    __device__ void sync() const { __syncwarp(); }
#else
    int lane() const { return 0; }
    uint32_t ballot(bool b) const { return b ? 1u : 0u; }
    double of(double v, int) const { return v; }
    void sync() const {}
#endif
};

// The density model in units of g_min.  x stands for ln(a / g_min) throughout.
struct TailModel {
    double rho, gamma;
    double body;      // 1 - 2 rho: mass below g_min
    double c1;        // 1 / (gamma - 1)
    double b;         // 1 - gamma / 3
    double ratio;     // (2 rho (gamma-1) / (1 - 2 rho))^(1/3): tail over body of p^(1/3) at g_min
    double ln_k;      // ln(2 rho s^2 / (gamma - 2)): alpha' is g_min exp(c1 ln_k)
    double ln_body;

    TQ_HD TailModel(double rho_, double gamma_, double s, uint32_t mode) : rho(rho_), gamma(gamma_) {
        body = 1.0 - 2.0 * rho;
        c1 = 1.0 / (gamma - 1.0);
        b = 1.0 - gamma / 3.0;
        ln_k = log(2.0 * rho * s * s / (gamma - 2.0));
        ln_body = mode == TQ_NONUNIFORM ? log(body) : 0.0;
        ratio = mode == TQ_NONUNIFORM ? cbrt(2.0 * rho * (gamma - 1.0) / body) : 0.0;
    }
    // Integral of p^(1/3) over [0, a] in units of its value at g_min: a / g_min up to g_min, then
    // 1 + ratio * (e^(b x) - 1) / b  (ratio * x for b = 0).
    TQ_HD double cuberoot_integral(double x) const {
        if (x <= 0.0) return exp(x);
        return 1.0 + ratio * (b == 0.0 ? x : expm1(b * x) / b);
    }
    // a / g_min at which cuberoot_integral reaches tau >= 0
    TQ_HD double cuberoot_integral_inverse(double tau) const {
        if (tau <= 1.0) return tau;
        const double rest = (tau - 1.0) / ratio;
        return b == 0.0 ? exp(rest) : exp(log1p(b * rest) / b);
    }
    // Right-hand side of the boxed alpha equations, F(x) = c1 (ln_k - ln Q(x)), and its derivative, for
    //   Q_U = mass inside (Section 4.1), and Q_N = (2 int p^(1/3))^3 / (2 a)^2 = body * I^3 * e^(-2x) (Section 4.2).
    TQ_HD double rhs(uint32_t mode, double x, double* slope) const {
        if (mode == TQ_UNIFORM) {
            if (x <= 0.0) { *slope = -c1; return c1 * (ln_k - log(body) - x); }
            const double z = 2.0 * rho * exp((1.0 - gamma) * x), q = 1.0 - z;
            *slope = -z / q;
            return c1 * (ln_k - log(q));
        }
        if (x <= 0.0) { *slope = -c1; return c1 * (ln_k - ln_body - x); }
        const double e = b == 0.0 ? 0.0 : expm1(b * x);
        const double i = 1.0 + ratio * (b == 0.0 ? x : e / b);
        *slope = c1 * (2.0 - 3.0 * ratio * (1.0 + e) / i);
        return c1 * (ln_k - ln_body - 3.0 * log(i) + 2.0 * x);
    }
};

constexpr int kSplitGrid = 128;
constexpr double kSplitFine = 1.4901161193847656e-08, kSplitCoarse = 2.384185791015625e-07;      // 2^-26, 2^-22: see close_in
constexpr double kSplitFirst = 9.094947017729282e-13, kSplitLnFirst = -27.72588722239781;   // 2^-40: the grid's first point, in place of 0
// k^-gamma at the grid points of one lane, k = j / 128 with j = t * kLanes + lane + 1: the same for every alpha, and for every
// record of one gamma.
template <class Lanes>
struct SplitGrid {
    double gamma = NAN, power[kSplitGrid / Lanes::kLanes];
    TQ_HD static double ln_k(int j) { return j < kSplitGrid ? log(static_cast<double>(j) / kSplitGrid) : kSplitLnFirst; }
    TQ_HD void prepare(const Lanes& lanes, double gamma_) {
        if (gamma == gamma_) return;
        gamma = gamma_;
#pragma unroll
        for (int t = 0; t < kSplitGrid / Lanes::kLanes; ++t) power[t] = exp(-gamma * ln_k(t * Lanes::kLanes + lanes.lane() + 1));
    }
};
TQ_HD inline int first_bit(uint64_t v) {                   // index of the lowest set bit
#ifdef __CUDA_ARCH__
    return __ffsll(static_cast<long long>(v)) - 1;
#else
    return __builtin_ctzll(v);
#endif
}

// The two-step quantizer's split (Appendix): k* = argmin_k Q_B(a, k) with
// Q_B^(1/3) = w^(1/3) (1-k)^(2/3) + u^(1/3) k^(2/3),  u = mass inside k a,  w = mass between k a and a.
struct Split {
    const TailModel& m;
    double x, a;                // a in units of g_min
    double outside, mass; // 2 rho a^(1-gamma), the mass beyond a; the mass inside
    TQ_HD Split(const TailModel& m_, double x_) : m(m_), x(x_), a(exp(x_)), outside(2.0 * m_.rho * exp((1.0 - m_.gamma) * x_)) {
        mass = x <= 0.0 ? m.body * a : 1.0 - outside;
    }

    TQ_HD double inner(double k, bool in_body) const {
        return in_body ? m.body * k * a : 1.0 - 2.0 * m.rho * exp((1.0 - m.gamma) * (x + log(k)));
    }
    // Negative where Q_B falls with k.  The derivative's sign is that of
    //     w^(2/3) (1-k)^(1/3) (u' k + 2 u)  -  u^(2/3) k^(1/3) (u' (1-k) + 2 w),      u' = du/dk,
    // whose terms are non-negative, so their cubes can be compared: the difference of the cubes has the same zeros.
    TQ_HD double slope(double k, double u, double du) const {
        double w = mass - u;
        if (w < 0.0) w = 0.0;
        const double p = du * k + 2.0 * u, q = du * (1.0 - k) + 2.0 * w;
        return w * w * (1.0 - k) * (p * p * p) - u * u * k * (q * q * q);
    }
    TQ_HD double slope_at(double k, double ln_k) const {
        if (k * a <= 1.0) return slope(k, m.body * k * a, m.body * a);
        const double beyond = 2.0 * m.rho * exp((1.0 - m.gamma) * x - m.gamma * ln_k);     // mass beyond k a, over k
        return slope(k, 1.0 - beyond * k, (m.gamma - 1.0) * beyond);
    }
    // Q_B(a, k), and d ln Q_B / dx along the minimum: at fixed k where k is a smooth minimum (its own motion does not
    // change Q_B to first order), along k = 1 / a where it is the kink.
    TQ_HD double factor(double k, bool kink, double* ln_slope) const {
        const bool in_body = k * a <= 1.0;
        const double u = kink ? m.body : inner(k, in_body);
        double w = mass - u;
        if (w < 0.0) w = 0.0;
        const double cw = cbrt(w * (1.0 - k) * (1.0 - k)), cu = cbrt(u * k * k), t = cw + cu;
        const double dmass = (m.gamma - 1.0) * (1.0 - mass);
        *ln_slope = kink ? (cw * dmass / w + 2.0 * (k * cw / (1.0 - k) - cu)) / t
                         : (in_body ? cw * (dmass - u) / w + cu : cw * (dmass - (m.gamma - 1.0) * (1.0 - u)) / w + cu * (m.gamma - 1.0) * (1.0 - u) / u) / t;
        return t * t * t;
    }
    // Q_B(a, 0) = Q_B(a, 1) = Q_U(a), so the minimum is a point where Q_B turns from falling to rising.  Every
    // such turn between neighbours of a 128-point grid is closed in on; the turn with the smallest Q_B wins.  No turn:
    // the minimum is an end.  Where the density jumps (k a = g_min) the turn may be a kink, which is tested for by itself.
    // Q_B is flat at a smooth turn: an error of 2^-24 there enters Q_B by its square, and the alpha iteration asks for no more (alpha, exponents 2.2 to 4.5,
    // against 64-bit significands: off by 2^-52 in the middle of 12000 cases, by 2^-45 in a tenth and by up to the 2^-40 at which it stops; with
    // the bracket closed in to the end 2^-50, 2^-44 and 2^-40).
    template <class Lanes>
    TQ_HD double best(const Lanes& lanes, const SplitGrid<Lanes>& grid, bool fine, double* q_best, double* ln_slope) const {
        constexpr int n = Lanes::kLanes;
        *ln_slope = NAN;
        if (x <= 0.0) { *q_best = mass; return 0.5; }            // flat density: Q_B is the same for every k
        uint64_t down[2] = {0, 0};                               // bit j - 1: Q_B falls at k = j / 128 (the end counts as rising)
        // (k a)^(1-gamma) as a product of powers, unless one of the two could leave the range of a double
        const bool powers = m.gamma * fmax(x, -kSplitLnFirst) < 600.0;
#pragma unroll
        for (int t = 0; t < kSplitGrid / n; ++t) {
            const int j = t * n + lanes.lane() + 1;               // the last place is the grid's first point
            const double k = j < kSplitGrid ? static_cast<double>(j) / kSplitGrid : kSplitFirst;
            const bool in_body = k * a <= 1.0;
            double beyond = outside * grid.power[t];            // mass beyond k a, over k
            if (!powers) beyond = 2.0 * m.rho * exp((1.0 - m.gamma) * x - m.gamma * grid.ln_k(j));
            const double u = in_body ? m.body * k * a : 1.0 - beyond * k;
            const bool falling = slope(k, u, in_body ? m.body * a : (m.gamma - 1.0) * beyond) < 0.0;
            down[t * n / 64] |= static_cast<uint64_t>(lanes.ballot(falling)) << (t * n % 64);
        }
        const uint64_t first = down[1] >> 63;
        down[1] &= ~(1ull << 63);
        uint64_t turns0 = ~down[0] & ((down[0] << 1) | first), turns1 = ~down[1] & ((down[1] << 1) | (down[0] >> 63));
        double best_k = 0.0, best_q = mass;
#pragma unroll 1
        while ((turns0 | turns1) != 0) {
            const int j = (turns0 ? first_bit(turns0) : 64 + first_bit(turns1)) + 1;
            if (turns0) turns0 &= turns0 - 1; else turns1 &= turns1 - 1;
            bool kink = false;
            const double k = close_in(lanes, j > 1 ? static_cast<double>(j - 1) / kSplitGrid : kSplitFirst, static_cast<double>(j) / kSplitGrid, fine, &kink);
            double slope;
            const double q = factor(k, kink, &slope);
            if (q < best_q) { best_q = q; best_k = k; *ln_slope = slope; }
        }
        *q_best = best_q;
        return best_k;
    }
    // Q_B falls at lo and does not at hi: the lanes' trial points cut the bracket into kLanes + 1 parts each time.  A warp's cubic through four of
    // them ends that; otherwise it goes on until the bracket is 2^-17 wide (relative), where the slope is close to a straight line whose zero
    // is off by the square of that width times a factor that grows where the slope bends; `fine` adds a Newton step with the slope of that line.
    // Against 64-bit significands, 18000 cases of exponents 2.05 to 10, alpha given or solved for, levels are off by 2^-48 to 2^-53 in the
    // middle of the cases and by up to 2^-33 (the rounding of the slope) either way to the end, the coarse split by up to 2^-24.
    template <class Lanes>
    TQ_HD double close_in(const Lanes& lanes, double lo, double hi, bool fine, bool* at_kink) const {
        constexpr int n = Lanes::kLanes;
        const double kink = 1.0 / a;
        if (kink > lo && kink < hi) {
            const double du_tail = 2.0 * m.rho * (m.gamma - 1.0) * a;
            const bool before = slope(kink, m.body, m.body * a) < 0.0, after = slope(kink, m.body, du_tail) < 0.0;
            if (before && !after) { *at_kink = true; return kink; }
            if (before) lo = kink; else hi = kink;
        }
        double s_lo = NAN, s_hi = NAN;                           // slopes at the ends, where known
#pragma unroll 1
        for (int it = 0; it < 64 && (hi - lo > 7.62939453125e-6 * hi || !(s_lo < 0.0) || !(s_hi >= 0.0)); ++it) {
            const double step = (hi - lo) * (1.0 / (n + 1));
            const double k = lo + step * (lanes.lane() + 1), s = slope_at(k, log(k));
            const uint32_t rises = lanes.ballot(!(s < 0.0));
            const int c = rises ? first_bit(rises) : n;            // trial points before the first one where Q_B rises
            if constexpr (n >= 8) {
                // Two trial points on either side of the turn: the zero of the cubic k(slope) through the four, if they are close enough for it.  How
                // close that is depends on where the slope bends (k near 0 or 1, large exponents): with r2 and r3 the second and third
                // differences over the first, the cubic is off by less than a quarter of the 3/2 power of max(r2^2, r3), in steps.  `fine` goes
                // on from there by the slope at that point, with its first and second derivative from the differences.
                if (c >= 2 && c <= n - 2) {
                    const double sa = lanes.of(s, c - 2), sb = lanes.of(s, c - 1), sc = lanes.of(s, c), sd = lanes.of(s, c + 1);
                    if (sa < sb && sb < sc && sc < sd) {
                        // Neville's scheme at slope 0, places counted from the first point in steps
                        const double ra = 1.0 / (sb - sa), rb = 1.0 / (sc - sb), rc = 1.0 / (sd - sc), rd = 1.0 / (sc - sa), re = 1.0 / (sd - sb), rf = 1.0 / (sd - sa);
                        const double ab = -sa * ra, bc = 1.0 - sb * rb, cd = 2.0 - sc * rc;
                        const double abc = (ab * sc - bc * sa) * rd, bcd = (bc * sd - cd * sb) * re;
                        const double at = (abc * sd - bcd * sa) * rf;
                        const double before = (sc - sb - (sb - sa)) * rb, after = (sd - sc - (sc - sb)) * rb;
                        const double bend = fmax(fmax(before * before, after * after), fabs(after - before)), most = (fine ? kSplitFine : kSplitCoarse) * lo;
                        if (at >= 1.0 && at <= 2.0 && bend * bend * bend * (step * step) <= most * most) {
                            double k = lo + step * (static_cast<double>(c - 1) + at);
                            if (fine) {
                                const double off = at - 1.5, mean = 0.5 * (before + after), third = after - before;
                                const double per_slope = rb / (1.0 + off * mean + (0.5 * off * off - 1.0 / 24.0) * third);
                                const double by = slope_at(k, log(k)) * per_slope;                  // steps
                                const double better = k - step * (by + 0.5 * by * by * (mean + off * third));
                                if (better > lo && better < hi) k = better;
                            }
                            return k;
                        }
                    }
                }
            }
            const double new_lo = c > 0 ? lo + step * c : lo, new_hi = c < n ? lo + step * (c + 1) : hi;
            if (c > 0) s_lo = lanes.of(s, c - 1);
            if (c < n) s_hi = lanes.of(s, c);
            if (!(new_hi - new_lo < hi - lo)) break;
            lo = new_lo; hi = new_hi;
        }
        if (!(s_lo < 0.0 && s_hi >= 0.0)) return 0.5 * (lo + hi);
        const double per_slope = (hi - lo) / (s_hi - s_lo);
        double k = lo - s_lo * per_slope;
        if (fine) {
            const double better = k - slope_at(k, log(k)) * per_slope;
            if (better > lo && better < hi) k = better;
        }
        return k;
    }
};

TQ_HD inline float ceil_to_float(double v) {
    float f = static_cast<float>(v);
    if (static_cast<double>(f) < v) f = nextafterf(f, 3.402823466e38f * 2.0f);   // towards +inf
    return f;
}

// inv_width / inv_step from a finished level table.  Rounded up so that a value sitting on the
// top level maps to probability >= 1 and is reproduced exactly.
template <class Lanes>
TQ_HD inline tq_status finish(const Lanes& lanes, tq_params_t* p) {
    const uint32_t s = p->num_levels - 1;
    bool bad = false;
    for (uint32_t k = lanes.lane(); k < s; k += Lanes::kLanes) {
        const float w = static_cast<float>(static_cast<double>(p->levels[k + 1]) - static_cast<double>(p->levels[k]));
        p->inv_width[k] = ceil_to_float(1.0 / static_cast<double>(w));
        if (!(p->levels[k + 1] > p->levels[k]) || !finite_f(p->inv_width[k])) bad = true;
    }
    const float alpha = p->levels[s], inv_step = ceil_to_float(static_cast<double>(s) / static_cast<double>(2.0f * alpha));
    if (lanes.lane() == 0) { p->alpha = alpha; p->inv_step = inv_step; }
    return lanes.ballot(bad) || !finite_f(inv_step) ? TQ_ERR_DEGENERATE_LEVELS : TQ_OK;
}

TQ_HD inline bool bits_for_levels(uint32_t num_levels, uint32_t* bits) {
    for (uint32_t b = 1; b <= 4; ++b)
        if ((1u << b) == num_levels) { *bits = b; return true; }
    return false;
}

TQ_HD inline void clear(tq_params_t* p) {
    p->bits = p->num_levels = p->mode = p->flags = 0;
    p->alpha = p->inv_step = p->gamma = p->g_min = p->rho = 0.0f;
    p->iterations = 0; p->reserved[0] = p->reserved[1] = 0.0f;
    for (int k = 0; k < TQ_MAX_LEVELS; ++k) { p->levels[k] = 0.0f; p->inv_width[k] = 0.0f; }
}

// The boxed alpha equation x = F(x), from x0 = ln(alpha' / g_min) until a plain step changes alpha by <= 1e-12
// relative.  The plain iteration converges linearly (70 steps for gamma = 3, s = 15).  F' comes with F, so a step goes to
// the root of the tangent of F(x) - x where that cannot change the outcome; x = F(x) is tested on the way in any case.  For the
// quantizers of Sections 4.1 and 4.2 and x > 0, every iterate is >= x0 because Q <= 1, and wherever F' < 1 it grows with x and
// stays below 1, so F - x is convex and falls: one fixed point, which no tangent from its left passes.
//   x0 > 0 and -0.9 <= F'(x0): no 2-cycle (F' > -1), so the plain iteration reaches that point too.  Its largest iterate is F(x0)
//   or the fixed point; it is stopped by max|g| exactly when one of the two is beyond, and either shows as a plain step beyond.
//   Elsewhere steps stay plain (the plain iteration may end in a 2-cycle, which is its result) but where F rises from x on
//   (F' >= 0, F(x) >= x): it then runs up to the point that the tangents approach from the same side.
// The two-step quantizer takes tangents wherever F' >= 0.  F has a kink at x = 0, which no tangent step crosses.  Stops when a plain
// step has passed max|g|.
template <class Lanes>
TQ_HD inline double solve_alpha(const Lanes& lanes, const SplitGrid<Lanes>& grid, const TailModel& m, uint32_t mode, double x_cap,
                                int* iterations) {
    double x = m.c1 * m.ln_k;
    double least = mode == TQ_BISCALED || !(x > 0.0) ? 0.0 : -0.9;      // smallest F' that a tangent step is taken at
    double x_before = 0.0, d_before = 0.0, inv_before = NAN;            // the iterate before, if a tangent step was taken there
    int it = 0;
    while (it < 10000 && !(x > x_cap)) {
        double slope, f;
        if (mode == TQ_BISCALED) {
            double q, ln_slope;
            Split(m, x).best(lanes, grid, false, &q, &ln_slope);
            f = m.c1 * (m.ln_k - log(q));
            slope = -m.c1 * ln_slope;
        } else {
            f = m.rhs(mode, x, &slope);
        }
        if (it == 0 && !(slope >= least)) least = 0.0;
        ++it;
        const double d = f - x, inv = 1.0 / (1.0 - slope);
        double root = f + d * slope * inv;                               // = x + d / (1 - slope)
        if (mode == TQ_BISCALED) {
            // the cubic x(F - x) through this iterate and the one before, with both tangents, once it lies well inside the last step
            const double width = d_before - d, t = -d / width;
            if (inv_before == inv_before && fabs(t) < 0.25) {
                const double u = 1.0 - t;
                root = x + t * (t * (3.0 - 2.0 * t) * (x_before - x) - width * u * (inv * u - inv_before * t));
            }
        }
        const bool same = mode == TQ_BISCALED || least < 0.0 || d >= 0.0;
        const bool take = same && slope >= least && slope < 0.999 && x > 0.0 && root > 0.0 && finite_d(root) && !(f > x_cap) && !(root > x_cap);
        x_before = x; d_before = d; inv_before = take ? inv : NAN;
        x = f;
        if (fabs(d) <= 1e-12) break;
        if (take) x = root;
    }
    *iterations = it;
    return x;
}

// Section 4 as a whole for one worker, by the lanes together.  Arguments are already range-checked; `out` is memory
// that all lanes see.
template <class Lanes>
TQ_HD inline tq_status design(const Lanes& lanes, SplitGrid<Lanes>& grid, const tq_stats_t* st, uint32_t num_levels, uint32_t bits, uint32_t mode, double gamma,
                              int rule, double alpha_user, tq_params_t* out) {
    const bool first = lanes.lane() == 0;
    if (first) {
        clear(out);
        out->bits = bits; out->num_levels = num_levels; out->mode = mode;
    }
    const double s = static_cast<double>(num_levels - 1);
    uint32_t flags = 0;

    if (gamma != gamma) {  // NaN: Section 5, gamma = 1 + n / sum ln(g_j / g_min)
        if (st->n_tail == 0 || !(st->sum_log_tail > 0.0)) return TQ_ERR_DOMAIN;
        gamma = 1.0 + static_cast<double>(st->n_tail) / st->sum_log_tail;
        flags |= TQ_FLAG_GAMMA_FROM_MLE;
    }
    if (!(gamma > 2.0) || !finite_d(gamma)) return TQ_ERR_DOMAIN;
    if (!(st->g_min > 0.0f) || !finite_f(st->g_min) || st->d == 0) return TQ_ERR_DOMAIN;
    const double rho = static_cast<double>(st->n_tail) / (2.0 * static_cast<double>(st->d));
    if (!(rho > 0.0) || !(rho < 0.5)) return TQ_ERR_DOMAIN;
    const double g_min = static_cast<double>(st->g_min);
    const TailModel m(rho, gamma, s, mode);
    if (mode == TQ_BISCALED) grid.prepare(lanes, gamma);
    int iterations = 0;

    double alpha;
    if (rule == TQ_ALPHA_USER) {
        if (!(alpha_user > 0.0) || !finite_d(alpha_user)) return TQ_ERR_DOMAIN;
        alpha = alpha_user;
    } else if (rule == TQ_ALPHA_MAXABS) {                    // Section 5 baselines: no truncation
        if (!(st->max_abs > 0.0f)) return TQ_ERR_DOMAIN;
        alpha = static_cast<double>(st->max_abs);
    } else {
        const double cap = static_cast<double>(st->max_abs);
        double x = m.c1 * m.ln_k;                            // alpha'
        if (rule == TQ_ALPHA_FIXED_POINT)
            x = solve_alpha(lanes, grid, m, mode, cap > 0.0 ? log(cap / g_min) : INFINITY, &iterations);
        alpha = g_min * exp(x);
        if (alpha != alpha) return TQ_ERR_DOMAIN;
        if (alpha < g_min) { alpha = g_min; flags |= TQ_FLAG_ALPHA_AT_GMIN; }
        if (cap > 0.0 && alpha > cap) { alpha = cap; flags |= TQ_FLAG_ALPHA_CAPPED; }
    }
    if (first) {
        out->gamma = static_cast<float>(gamma); out->g_min = st->g_min; out->rho = static_cast<float>(rho);
        out->iterations = iterations; out->flags = flags;
    }

    const float alpha_f = static_cast<float>(alpha);
    if (!(alpha_f > 0.0f) || !finite_f(2.0f * alpha_f)) return TQ_ERR_DOMAIN;
    const double a = static_cast<double>(alpha_f);
    const uint32_t si = num_levels - 1;
    lanes.sync();                                            // the cleared record
    if (mode == TQ_UNIFORM) {
        const double step = 2.0 * a / s;                     // Section 4.1 codebook
        for (uint32_t k = 1 + lanes.lane(); k < si; k += Lanes::kLanes) out->levels[k] = static_cast<float>(-a + static_cast<double>(k) * step);
    } else if (mode == TQ_BISCALED) {
        // Appendix: density s c_in / D inside k* alpha and s c_out / D outside, c = (mean density)^(1/3),
        // D = 2 alpha (c_out (1 - k*) + c_in k*).  Level k sits where the density accumulated from the
        // centre reaches k - s/2.  Upper half, then mirrored.
        const Split split(m, log(a / g_min));
        double q, ln_slope;
        const double k = split.best(lanes, grid, true, &q, &ln_slope), beta = k * a;
        const double u = k > 0.0 ? split.inner(k, k * split.a <= 1.0) : 0.0;
        const double c_in = cbrt(u / (2.0 * beta));
        const double c_out = cbrt((split.mass - u) / (2.0 * (a - beta)));
        const double denom = 2.0 * a * (c_out * (1.0 - k) + c_in * k);
        const double lam_in = s * c_in / denom, lam_out = s * c_out / denom;
        for (uint32_t j = (si + 1) / 2 + lanes.lane(); j < si; j += Lanes::kLanes) {
            const double c = static_cast<double>(j) - 0.5 * s;
            const double x = c <= lam_in * beta ? c / lam_in : beta + (c - lam_in * beta) / lam_out;
            out->levels[j] = static_cast<float>(x);
            out->levels[si - j] = -static_cast<float>(x);
        }
    } else {
        // lambda_s = s p^(1/3) / int p^(1/3): level k sits where the running integral of p^(1/3)
        // from the centre reaches (2k/s - 1) of its value at alpha.  Upper half, then mirrored.
        const double total = m.cuberoot_integral(log(a / g_min));
        for (uint32_t k = (si + 1) / 2 + lanes.lane(); k < si; k += Lanes::kLanes) {
            const double tau = (2.0 * static_cast<double>(k) / s - 1.0) * total;
            const float l = static_cast<float>(g_min * m.cuberoot_integral_inverse(tau));
            out->levels[k] = l;
            out->levels[si - k] = -l;
        }
    }
    if (first) { out->levels[0] = -alpha_f; out->levels[si] = alpha_f; }
    lanes.sync();
    return finish(lanes, out);
}

static bool valid_request(uint32_t num_levels, int mode, int rule, uint32_t* bits) {
    if (!bits_for_levels(num_levels, bits)) return false;
    if (mode != TQ_UNIFORM && mode != TQ_NONUNIFORM && mode != TQ_BISCALED) return false;
    return rule == TQ_ALPHA_CLOSED || rule == TQ_ALPHA_FIXED_POINT || rule == TQ_ALPHA_USER || rule == TQ_ALPHA_MAXABS;
}

// One warp per worker.  A worker whose statistics are outside the model's domain gets
// flags = TQ_FLAG_INVALID, iterations = the status code, alpha = 0 and an all-zero codebook.
// One kernel per quantizer: a record runs straight through code that is fetched for the first time, so its length counts
// (all three in one kernel: 18.2 us instead of 7.7 us for 4 workers, non-uniform, 8 levels).
constexpr int kParamsWarps = 4;
template <uint32_t MODE>
__global__ void __launch_bounds__(32 * kParamsWarps)
params_kernel(const tq_stats_t* stats, uint32_t n, uint32_t num_levels, uint32_t bits, double gamma, int rule,
              double alpha_user, tq_params_t* out) {
    __shared__ tq_params_t s_p[kParamsWarps];
    const uint32_t warp = threadIdx.x >> 5, i = blockIdx.x * kParamsWarps + warp;
    if (i >= n) return;              // nothing of this warp reads or writes memory
    const OneWarp lanes;
    tq_params_t* p = &s_p[warp];
    SplitGrid<OneWarp> grid;
    if (MODE == TQ_BISCALED && gamma == gamma) grid.prepare(lanes, gamma);      // while the statistics are still being taken
    pdl_wait();
    const tq_stats_t st = stats[i];
    const tq_status s = design(lanes, grid, &st, num_levels, bits, MODE, gamma, rule, alpha_user, p);
    __syncwarp();
    if (s != TQ_OK && lanes.lane() == 0) {
        clear(p);
        p->bits = bits; p->num_levels = num_levels; p->mode = MODE;
        p->flags = TQ_FLAG_INVALID; p->iterations = static_cast<int32_t>(s);
    }
    __syncwarp();
    const uint32_t* from = reinterpret_cast<const uint32_t*>(p);
    uint32_t* to = reinterpret_cast<uint32_t*>(out + i);
    for (uint32_t w = lanes.lane(); w < sizeof(tq_params_t) / 4; w += 32) to[w] = from[w];
}

cudaError_t launch_params_device(const tq_stats_t* stats_dev, uint32_t n, uint32_t num_levels, uint32_t bits, uint32_t mode,
                                 double gamma, int rule, double alpha_user, tq_params_t* params_dev, cudaStream_t stream) {
    const uint32_t warps = n < kParamsWarps ? n : kParamsWarps;      // few records: no idle warps to launch
    const dim3 grid((n + kParamsWarps - 1) / kParamsWarps);
    auto* kernel = mode == TQ_UNIFORM ? params_kernel<TQ_UNIFORM> : mode == TQ_NONUNIFORM ? params_kernel<TQ_NONUNIFORM> : params_kernel<TQ_BISCALED>;
    return launch_kernel(kernel, grid, 32 * warps, 0, stream, stats_dev, n, num_levels, bits, gamma, rule, alpha_user, params_dev);
}

bool params_request_ok(uint32_t num_levels, int mode, int rule, uint32_t* bits) { return valid_request(num_levels, mode, rule, bits); }

}  // namespace tq

extern "C" tq_status tq_params_from_levels(const float* levels_host, uint32_t num_levels, tq_mode mode,
                                           tq_params_t* out) {
    uint32_t bits = 0;
    if (!levels_host || !out || !tq::bits_for_levels(num_levels, &bits)) return TQ_ERR_INVALID_ARG;
    if (mode != TQ_UNIFORM && mode != TQ_NONUNIFORM && mode != TQ_BISCALED) return TQ_ERR_INVALID_ARG;
    tq::clear(out);
    out->bits = bits; out->num_levels = num_levels; out->mode = mode;
    for (uint32_t k = 0; k < num_levels; ++k) out->levels[k] = levels_host[k];
    const float top = levels_host[num_levels - 1];
    if (!(top > 0.0f) || !tq::finite_f(2.0f * top) || levels_host[0] != -top) return TQ_ERR_DOMAIN;
    return tq::finish(tq::OneThread(), out);
}

extern "C" tq_status tq_params(const tq_stats_t* st, uint32_t num_levels, tq_mode mode, double gamma,
                               tq_alpha_rule rule, double alpha_user, tq_params_t* out) {
    uint32_t bits = 0;
    if (!st || !out || !tq::valid_request(num_levels, mode, rule, &bits)) return TQ_ERR_INVALID_ARG;
    tq::SplitGrid<tq::OneThread> grid;
    return tq::design(tq::OneThread(), grid, st, num_levels, bits, mode, gamma, rule, alpha_user, out);
}

extern "C" tq_status tq_params_batch(const tq_stats_t* st, uint32_t n_workers, uint32_t num_levels, tq_mode mode,
                                     double gamma, tq_alpha_rule rule, double alpha_user, tq_params_t* out) {
    uint32_t bits = 0;
    if (!st || !out || n_workers == 0 || n_workers > TQ_MAX_WORKERS) return TQ_ERR_INVALID_ARG;
    if (!tq::valid_request(num_levels, mode, rule, &bits)) return TQ_ERR_INVALID_ARG;
    tq::SplitGrid<tq::OneThread> grid;
    for (uint32_t i = 0; i < n_workers; ++i)
        if (tq_status s = tq::design(tq::OneThread(), grid, st + i, num_levels, bits, mode, gamma, rule, alpha_user, out + i)) return s;
    return TQ_OK;
}

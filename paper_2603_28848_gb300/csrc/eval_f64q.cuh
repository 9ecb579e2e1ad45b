// FP64 sample loop with an FP32 screen.
//
// FP64 runs at 1/64 of the FP32 rate on this GPU: one FP64 operation of a warp
// takes an SM partition's pipe for 64 cycles, about 300 of them per 2 -> 2
// sample, so the plain FP64 loop is bound by that pipe alone (1.6e9 samples/s).
// Most samples, though, lie so far from the energy shell that the Gaussian of
// Eq. (11) is zero in FP64, or too small to change any result.  So every
// sample is first screened in FP32 (Philox words, map, momenta, energy
// balance with a bound on its error), the samples that can matter are queued
// per warp as their Philox words, and 32 queued samples at a time are
// evaluated from scratch in FP64 on a full warp.
//
// What the screen drops, in terms of an upper bound L of log2 |w_n|:
//   * samples whose Gaussian exponent is below -1100 (|dE| > 39 sigma): their
//     FP64 weight is exactly 0 (2^-1075 is the smallest subnormal);
//   * samples with L < log2(largest |w_n| this warp has evaluated in the
//     segment) - kDropBits - log2 N, kDropBits = 66, N the task's samples.  L
//     takes the kinematic factors and the statistical ones from FP32 with their
//     rounding bounded (a few bits).  All such samples together are below 2^-66
//     of one that was summed, 2^-13 of the last place of the sum of w (and of
//     w^2 far below), and an increment holding nothing else has a share of w^2
//     below the 1e-30 = 2^-100 that the refinement counts as empty.
// A sample whose FP32 quantities leave the normal range is kept.
//
// Measured per sweep on trained maps, plain loop -> this one: MB 2 -> 2, 32
// points, 1e5 x 2 samples: 8.28 -> 0.77 ms; BE 2 -> 2, 2 species, 128 points,
// 1e5 x 2: 55.2 -> 9.5 ms (up to 40% of the samples are evaluated, the FP64 pipe
// is 79% busy, about 120 operations per queued sample).
#pragma once

#include "math_table.cuh"

namespace best {

constexpr float kDropBits = 66.0f;

// ---- FP64 elementary functions of this loop: fewer FP64 operations than the
// library's, at the price of a restricted range (checked or falling back), and
// no larger an error.  Measured against 112-bit arithmetic at 4e5 points, root
// mean square and largest error in units of the last place, the library's in
// brackets: 1/sqrt 0.289, 0.500 (0.289, 0.507); sin 0.305, 1.25 (0.337, 1.31)
// and cos 0.305, 1.49 (0.364, 1.35) over [-pi, pi]; 2^x 0.289, 0.537 (0.302,
// 0.847) over [-1000, 0]. ----

// The float next to a positive double in float range, towards zero, and back:
// integer operations only (FP64 conversions use the FP64 pipe).
__device__ __forceinline__ float trunc_f32(double x) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
    return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
}
__device__ __forceinline__ double widen_f32(float x) {        // positive normal float, exact
    const uint32_t b = __float_as_uint(x);
    return __hiloint2double(static_cast<int>((b >> 3) + 0x38000000u), static_cast<int>(b << 29));
}
__device__ __forceinline__ double flip_sign(double x, uint32_t mask) {
    return __hiloint2double(__double2hiint(x) ^ static_cast<int>(mask), __double2loint(x));
}

// 1/sqrt(x): FP32 estimate y (22 bits) and one step of Halley's third-order
// iteration (relative error 5/16 e^3 < 2^-60 before rounding).  y has 24 bits:
// y^2 is exact, so that 1 - x y^2 carries no rounding of the size of x y^2.
__device__ __forceinline__ double rsqrt_halley(double x) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(x));
    if (hi - 0x39000000u > 0x0DFFFFFFu) return rsqrt(x);      // outside [2^-111, 2^113): zero, subnormal, huge, NaN
    const double y = widen_f32(rsqrt_ftz(trunc_f32(x)));
    const double e = fma(-x, y * y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}

// sin and cos of |x| <= pi: the nearest a_k = k pi / 128 of the table, the
// Taylor polynomials of r = |x| - a_k (|r| <= pi / 256, the difference is
// exact) and the addition theorem (table-driven reduction after Gal and Tang).
// The polynomials' tails, 1/120 - r^2/5040 and 1/24 - r^2/720, are FP32 numbers:
// their rounding enters with r^4 < 2.3e-8, below 2^-53 of the results.
__device__ __forceinline__ void sincos_table(double x, const double* tab, double* s, double* c) {
    const uint32_t sign = static_cast<uint32_t>(__double2hiint(x)) & 0x80000000u;
    const double ax = flip_sign(x, sign);
    // (below 2^-126: k = 0)
    const uint32_t hx = static_cast<uint32_t>(__double2hiint(ax));
    const float xf = hx < 0x38100000u ? 0.0f : trunc_f32(ax);
    const int k = min(__float2int_rn(xf * 40.743665431525206f), kTrigEntries - 1);      // 128 / pi
    const double* T = tab + 5 * k;
    const double a = T[0], S = T[1], C = T[2];
    const double r = ax - a;
    const double r2 = r * r;
    const float rf = static_cast<uint32_t>(__double2hiint(r2)) < 0x38100000u ? 0.0f : trunc_f32(r2);
    const double p5 = widen_f32(fmaf(rf, -1.0f / 5040.0f, 1.0f / 120.0f));
    const double p4 = widen_f32(fmaf(rf, -1.0f / 720.0f, 1.0f / 24.0f));
    const double sr = fma(r * r2, fma(r2, p5, -1.0 / 6.0), r);
    const double cm = r2 * fma(r2, p4, -0.5);
    *s = flip_sign(S + fma(C, sr, fma(S, cm, T[3])), sign);
    *c = C + fma(-S, sr, fma(C, cm, T[4]));
}

// 2^x, x <= 0: 2^k 2^(j/32) 2^r, |r| <= 1/64, Taylor polynomial of 2^r - 1.
__device__ __forceinline__ double exp2_table(double x, const double* tab) {
    // hi word of x: beyond -1000 (or NaN) the library's function, which handles subnormal results
    if (static_cast<uint32_t>(__double2hiint(x)) - 0x80000000u > 0x408F4000u - 1u) return exp2(x);
    const uint32_t hx = static_cast<uint32_t>(__double2hiint(x)) & 0x7fffffffu;
    const float xf = hx < 0x38100000u ? 0.0f : trunc_f32(flip_sign(x, 0x80000000u));    // |x|
    const int n = __float2int_rn(xf * 32.0f);
    // n / 32 as a double (0 for n = 0)
    const double nd = n == 0 ? 0.0 : widen_f32(static_cast<float>(n) * 0.03125f);
    const double r = x + nd;
    double p = fma(r, 0x1.430912f86c787p-13, 0x1.5d87fe78a6731p-10);       // ln(2)^k / k!
    p = fma(r, p, 0x1.3b2ab6fba4e77p-7);
    p = fma(r, p, 0x1.c6b08d704a0c0p-5);
    p = fma(r, p, 0x1.ebfbdff82c58fp-3);
    p = fma(r, p, 0x1.62e42fefa39efp-1);
    const int k = -n;                                                     // x = k/32 + r
    const double* T = tab + 5 * kTrigEntries + 2 * (k & 31);
    const double v = fma(T[0], fma(p, r, T[1]), T[0]);
    return __hiloint2double(__double2hiint(v) + ((k >> 5) << 20), __double2loint(v));
}

// A product of doubles as a 64-bit significand m in [2^63, 2^64) and an
// exponent, value m / 2^63 2^e: a multiplication is a 64 x 64 -> high 64-bit
// integer product (about 16 issue slots instead of the 64 cycles an FP64
// multiplication takes the pipe) and loses at most 2^-62 (FP64: 2^-53).  It
// neither overflows nor underflows before value().  Of zeros and normal
// numbers: an infinite factor, a NaN or, where it is looked for (mul_f), a
// subnormal one sets rare, and the product is to be taken with
// multiplications.  (With all of those handled in place the MB sweep took
// 0.84 to 0.875 instead of 0.81 ms.)
struct Product {
    uint64_t m;
    int e;
    uint32_t sign;          // bit 31
    bool zero, rare;
    __device__ __forceinline__ explicit Product(double x) : m(1ull << 63), e(0), sign(0), zero(false), rare(false) { mul_f(x); }
    __device__ __forceinline__ void mul(double x) {
        const uint64_t b = static_cast<uint64_t>(__double_as_longlong(x));
        const int ex = static_cast<int>((b >> 52) & 0x7FF);
        sign ^= static_cast<uint32_t>(b >> 32);
        zero |= ex == 0;
        rare |= ex == 0x7FF;
        const uint64_t h = __umul64hi(m, (b << 11) | (1ull << 63));
        const int up = static_cast<int>(h >> 63);
        m = h << (1 - up);
        e += ex - 1023 + up;
    }
    __device__ __forceinline__ void mul_f(double x) {
        const uint32_t hi = static_cast<uint32_t>(__double2hiint(x));
        rare |= (hi & 0x7FF00000u) == 0u && ((hi << 1) | static_cast<uint32_t>(__double2loint(x))) != 0u;
        mul(x);
    }
    __device__ __forceinline__ double value() const {
        uint64_t t = m + 0x400;                     // rounded to 53 bits
        int x = e;
        if (t < m) {
            t = 1ull << 63;
            ++x;
        }
        const uint32_t sg = sign & 0x80000000u;
        if (zero || x < -1100) return 0.0;
        if (x < -1022 || x > 1023) return flip_sign(scalbn(static_cast<double>(t >> 11), x - 52), sg);
        return flip_sign(__longlong_as_double(static_cast<long long>((static_cast<uint64_t>(x + 1023) << 52) |
                                                                     ((t >> 11) & 0x000FFFFFFFFFFFFFull))), sg);
    }
};

// a < b for doubles neither of which is NaN, as integers (an FP64 comparison
// takes the FP64 pipe): b > 0; a negative a compares less.
__device__ __forceinline__ bool less_pos(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b);
}

// Cubic spline value at comoving q inside [q_0, q_{n-1}], the interval from
// FP32 (a guess within one interval, as in spline_eval).  On an evenly spaced
// grid the distance from q_0 is taken in FP64 first, as there: a grid far from
// zero is narrower than FP32 resolves.
__device__ __forceinline__ double spline64(const double* coef, const double* knots, double q, const Geometry& g,
                                           float inv_step, double q0, float lq0_step) {
    float x;
    if (g.log_spaced) {
        x = fmaf(lg2_ftz(trunc_f32(q)), inv_step, -lq0_step);
    } else {
        const double d = (q - q0) * g.inv_step;
        x = static_cast<uint32_t>(__double2hiint(d)) < 0x38100000u ? 0.0f : trunc_f32(d);      // (below 2^-126: 0)
    }
    int j = static_cast<int>(x);
    j = min(max(j, 0), g.n_grid - 2);
    const double t = q - knots[j];
    const double2* cp = reinterpret_cast<const double2*>(coef) + 2 * j;
    const double2 lo = cp[0], hi = cp[1];
    const double f = fma(fma(fma(hi.y, t, hi.x), t, lo.y), t, lo.x);
    return __double2hiint(f) < 0 ? 0.0 : f;
}

// Weight of one sample in FP64 (kin_at and stat_at of eval_impl.cuh, the same
// formulas) with the functions above; dy: the mapped increments' widths; C
// lives in shared memory.  rare: some factor is subnormal, infinite or a NaN,
// and the weight is plain_weight64's.
template <int NLEG>
__device__ __forceinline__ double weight64(const SegConst<double, NLEG>& C, const double* y, const double* dy,
                                           const double* s_spline, const double* knots, const Geometry& g,
                                           const SegSetup<float, NLEG>& s32, double q0, double qN, int ncoef,
                                           const double* tab, bool* rare) {
    constexpr int NI = NLEG - 2;
    double px = 0.0, py = 0.0, pz = C.pobs_sig;
    double bal = C.sgn_obs_E;
    double Esum = C.e_obs;
    Product w(C.c0);
    const bool scaled = C.inv_a != 1.0;
    bool cut = false;
#pragma unroll
    for (int j = 0; j < NI; ++j) {
        const double r = y[3 * j];
        double st, ct, sp, cp;
        sincos_table(y[3 * j + 1], tab, &st, &ct);
        sincos_table(y[3 * j + 2], tab, &sp, &cp);             // angle phi - pi
        const uint32_t sg = static_cast<uint32_t>(__double2hiint(C.sig[j])) & 0x80000000u;
        const double p = scaled ? r * C.inv_a : r;
        const double nps = flip_sign(p * st, sg ^ 0x80000000u);     // cos(phi) = -cos(phi - pi)
        px = fma(nps, cp, px);
        py = fma(nps, sp, py);
        pz = fma(flip_sign(p, sg), ct, pz);
        const double E2 = fma(p, p, C.m2[j]);
        const double rE = rsqrt_halley(E2);
        const double E = E2 * rE;
        cut |= less_pos(E, C.e_cut);
        bal += flip_sign(E, static_cast<uint32_t>(__double2hiint(C.sgnE[j])) & 0x80000000u);
        if (C.frac) Esum += E;
        w.mul(dy[3 * j]);
        w.mul(dy[3 * j + 1]);
        w.mul(dy[3 * j + 2]);
        w.mul(r);
        w.mul(r);
        w.mul(st);
        w.mul(rE);
        if (C.cb[j] != 0.0) {                       // (0: 1 + eta f of a Maxwell-Boltzmann leg, 1)
            double f = spline64(s_spline + C.spc[j] * ncoef, knots, r, g, s32.inv_step, q0, s32.lq0_step);
            if (C.fd[j]) f = f < 1.0 ? f : 1.0;
            w.mul_f(C.ca[j] != 0.0 ? fma(C.cb[j], f, C.ca[j]) : f);
        }
    }
    const double pc2 = fma(px, px, fma(py, py, pz * pz));
    double rpc, rEc, Ec;
    if (C.m2c == 0.0) {
        rEc = rsqrt_halley(less_pos(0.0, pc2) ? pc2 : 1e-30);
        Ec = pc2 * rEc;
        rpc = less_pos(0.0, pc2) ? rEc : 0.0;
    } else {
        const double Ec2 = pc2 + C.m2c;
        rEc = rsqrt_halley(Ec2);
        Ec = Ec2 * rEc;
        rpc = 0.0;
        if (C.cbc != 0.0 && less_pos(0.0, pc2)) rpc = rsqrt_halley(pc2);
    }
    cut |= less_pos(Ec, C.e_cut);
    bal += flip_sign(Ec, static_cast<uint32_t>(__double2hiint(C.sgn_cons)) & 0x80000000u);
    w.mul(rEc);
    // 2^x; where that is subnormal, and before, 2^512 of it goes into the exponent
    auto gauss = [&](double x) {
        const bool far = static_cast<uint32_t>(__double2hiint(x)) > 0xC08F4000u;     // x < -1000
        if (far) {
            x += 512.0;
            w.e -= 512;
        }
        return exp2_table(x, tab);
    };
    if (C.frac) {
        Esum += Ec;
        const double iS = 1.0 / Esum;
        const double x = bal * iS;
        w.mul(gauss(C.gauss_k * x * x));
        w.mul(2.0 * C.e_obs * iS);
    } else {
        w.mul(gauss(C.gauss_k * bal * bal));
    }
    if (C.cbc != 0.0) {
        double qc = pc2 * rpc;
        if (scaled) qc *= C.a;
        double fc;
        const bool below = less_pos(qc, q0), above = less_pos(qN, qc);
        if (!below && !above) {
            fc = spline64(s_spline + C.sp_cons * ncoef, knots, qc, g, s32.inv_step, q0, s32.lq0_step);
        } else {
            const double x = below ? C.tlo_a + C.tlo_b * Ec : C.thi_a + C.thi_b * Ec;
            const double den = C.eta_c == 1.0 ? expm1(x) : exp(x) - C.eta_c;
            fc = den > 0.0 ? 1.0 / den : 0.0;
        }
        if (C.fd_c) fc = fc < 1.0 ? fc : 1.0;
        w.mul_f(C.cac != 0.0 ? fma(C.cbc, fc, C.cac) : fc);
    }
    *rare = w.rare;
    return cut ? 0.0 : w.value();
}

// VEGAS map of one 52-bit uniform u = (k + 1/2) 2^-52 from its Philox words,
// table: the dimension's increments.  The increment and the fraction are those
// of t = u nb rounded to FP64, as every other evaluation of the same stream
// takes them (the fraction's rounding, 2^-48 for 50 increments, is the largest
// one before the energy balance: without it the samples are other ones by that
// much).  In integer operations: t = m 2^-53, rounded to nearest even at bit s.
__device__ __forceinline__ Real2<double> map_point64(uint32_t x0, uint32_t x1, int nb, const Real2<double>* table,
                                                     double* y, uint32_t* bin = nullptr) {
    const uint64_t k = (static_cast<uint64_t>(x0 >> 6) << 26) | (x1 >> 6);
    uint64_t m = (2 * k + 1) * static_cast<uint32_t>(nb);      // < 2^61
    const int s = max(0, 11 - __clz(static_cast<int>(m >> 32)));          // bits past the 53rd: 0 .. 8
    const uint32_t ulp = 1u << s;
    const uint32_t even = s ? ((static_cast<uint32_t>(m) >> s) & 1u) : 1u;
    m = (m + ((ulp >> 1) - 1u + even)) & ~static_cast<uint64_t>(ulp - 1u);
    uint32_t b = static_cast<uint32_t>(m >> 53);
    uint64_t frac = m & ((1ull << 53) - 1);                    // exact in FP64
    if (b == static_cast<uint32_t>(nb)) {                      // t rounded up to nb: the end of the last increment
        --b;
        frac = 1ull << 53;
    }
    const int lz = __clzll(static_cast<long long>(frac));
    const uint64_t bits = (((frac << lz) >> 11) & 0x000FFFFFFFFFFFFFull) | (static_cast<uint64_t>(1033 - lz) << 52);
    const double fr = __longlong_as_double(frac ? static_cast<long long>(bits) : 0);
    const Real2<double> e = table[b];
    *y = fma(e.dy, fr, e.y0);
    if (bin) *bin = b;
    return e;
}

// The weight of the queued sample whose words start at q, in the plain loop's
// arithmetic.
template <int NLEG>
__device__ __noinline__ double plain_weight64(const uint32_t* q, int nb, const Real2<double>* s_map,
                                              const SegSetup<double, NLEG>* S, const double* s_spline, int n_grid,
                                              int n_species, int log_spaced) {
    constexpr int D = 3 * (NLEG - 2);
    double y[D], jac = 1.0;
#pragma unroll
    for (int d = 0; d < D; ++d)
        jac *= map_point64(q[(2 * d) * kQueueSlots], q[(2 * d + 1) * kQueueSlots], nb, s_map + d * nb, &y[d]).dy;
    const int ncoef = 4 * (n_grid - 1);
    Geometry g{};
    g.n_grid = n_grid;
    g.log_spaced = log_spaced;
    return weight_at<double, NLEG, false>(S->C, y, jac, s_spline, s_spline + n_species * ncoef, g, S->inv_step, S->q0,
                                          S->lq0_step, S->qN, ncoef);
}

// The same in FP32 from the uniform's first 32 bits.  The 20 bits left out, and
// FP64's rounding, can take the point over an increment's edge: the mapped point
// is continuous there, the increment's width is not.  near_edge of the largest
// fraction says whether any may have crossed (nb 2^-32 of the samples per
// dimension).  Returns the increment's width.
__device__ __forceinline__ float map_point32(uint32_t x0, uint32_t x1, int nb, const Real2<float>* table, float* y,
                                             uint32_t* frac) {
    const uint32_t x = (x0 & ~63u) | (x1 >> 26);
    const uint64_t m = static_cast<uint64_t>(x) * static_cast<uint32_t>(nb);
    const Real2<float> e = table[static_cast<uint32_t>(m >> 32)];
    *frac = static_cast<uint32_t>(m);
    *y = fmaf(e.dy, static_cast<float>(static_cast<uint32_t>(m)) * 2.3283064365386963e-10f, e.y0);
    return e.dy;
}
__device__ __forceinline__ bool near_edge(uint32_t frac, int nb) { return frac >= 0u - static_cast<uint32_t>(nb); }

// log2 of an upper bound of |ca + cb f| at comoving q inside the grid: the FP32
// spline value plus its rounding bound (2^-18 of its terms' magnitudes); +inf or
// a NaN, either of which keeps the sample, where FP32 coefficients overflowed.
__device__ __forceinline__ float log2_factor_bound(const float* coef, const float* knots, float q, const Geometry& g,
                                                   float inv_step, float q0, float lq0_step, float ca) {
    int j = static_cast<int>(g.log_spaced ? fmaf(lg2_ftz(q), inv_step, -lq0_step) : (q - q0) * inv_step);
    j = min(max(j, 0), g.n_grid - 2);
    const float t = q - __ldg(knots + j);
    const float4 c = __ldg(reinterpret_cast<const float4*>(coef) + j);
    const float f = fmaf(fmaf(fmaf(c.w, t, c.z), t, c.y), t, c.x);
    const float at = fabsf(t);
    const float size = fmaf(fmaf(fmaf(fabsf(c.w), at, fabsf(c.z)), at, fabsf(c.y)), at, fabsf(c.x));
    // (at least 1e-36: FP32 subnormals flush to 0; the size, not f, carries what is not finite through)
    return lg2_ftz(ca + fmaxf(f, 0.0f) + fmaf(3.8e-6f, size, 1e-36f));
}

// Upper bound of log2 |w_n| of a sample from FP32 arithmetic, y the mapped
// point and jac the map's Jacobian; gauss gets an upper bound of the
// Gaussian's exponent.  Errors: a radius carries 2^-22 of itself and, from the
// 32-bit uniform, up to 2^-24 of the largest increment (1.2e-7 q_max); an angle
// and sin.approx / cos.approx 2^-20 absolute.  Every momentum component is then
// within 4e-6 of the momenta plus 1e-6 q_max / a of the four radii, and 4e-5 of
// the energies' sum plus that covers the balance ten times.  +inf where a
// factor leaves the normal range (or is not a number) or the conserved leg's
// energy is not resolved.  WEIGHT false: gauss alone.
template <int NLEG, bool WEIGHT>
__device__ __forceinline__ float log2_weight_bound(const SegSetup<float, NLEG>& S, const EvalParams& P, const float* y,
                                                   float jac, float* gauss) {
    constexpr int NI = NLEG - 2;
    const SegConst<float, NLEG>& C = S.C;
    const Geometry& g = P.geo;
    float px = 0.0f, py = 0.0f, pz = C.pobs_sig;
    float bal = C.sgn_obs_E, Esum = C.e_obs;
    float prod = jac;
#pragma unroll
    for (int j = 0; j < NI; ++j) {
        const float r = y[3 * j];
        float st, ct, sp, cp;
        __sincosf(y[3 * j + 1], &st, &ct);
        __sincosf(y[3 * j + 2], &sp, &cp);
        const float p = r * C.inv_a;
        const float nps = -C.sig[j] * (p * st);
        px = fmaf(nps, cp, px);
        py = fmaf(nps, sp, py);
        pz = fmaf(C.sig[j] * p, ct, pz);
        const float E2 = fmaf(p, p, C.m2[j]);
        const float rE = rsqrt_ftz(E2);
        const float E = E2 * rE;
        bal = fmaf(C.sgnE[j], E, bal);
        Esum += E;
        const float ru = fmaf(1.2e-7f, S.qN, r);
        prod *= ru * ru * (st + 2e-6f) * rE;
    }
    const float pc2 = fmaf(px, px, fmaf(py, py, pz * pz));
    const float Ec2 = pc2 + C.m2c;
    const float rEc = rsqrt_ftz(Ec2);
    const float Ec = Ec2 * rEc;
    bal = fmaf(C.sgn_cons, Ec, bal);
    Esum += Ec;
    prod *= rEc;
    // (no bound from a Gaussian whose factor FP32 does not hold: infinite error)
    const float err = fmaf(4e-5f, Esum, C.gauss_k > -1e37f ? 1e-6f * S.qN * C.inv_a : __int_as_float(0x7f800000));
    float d = fmaxf(fabsf(bal) - err, 0.0f);
    if (!(Esum < 1e30f)) d = 0.0f;                       // (overflowed, or not a number)
    float extra = 0.0f;
    if (C.frac) {
        const float iS = __fdividef(1.0f, Esum);
        d *= iS;
        extra = lg2_ftz(2.0f * C.e_obs * iS);
    }
    const float e = C.gauss_k * d * d;
    *gauss = e;
    if constexpr (!WEIGHT) return 0.0f;
    if (!(prod > 1e-37f && prod < 1e37f && Ec > 4.0f * err)) return __int_as_float(0x7f800000);
    const float kin = lg2_ftz(prod) + extra + e;
    // the statistical factors, 1 + f or f of every leg (|ca + cb f| is at most ca + f)
    const int ncoef = 4 * (g.n_grid - 1);
    float stat = 0.0f;
#pragma unroll
    for (int j = 0; j < NI; ++j)
        stat += log2_factor_bound(P.coef32 + C.spc[j] * ncoef, P.knots32, y[3 * j], g, S.inv_step, S.q0, S.lq0_step,
                                  C.ca[j]);
    const float qc = sqrtf(pc2) * C.a;
    if (qc > S.q0 && qc < S.qN) {
        stat += log2_factor_bound(P.coef32 + C.sp_cons * ncoef, P.knots32, qc, g, S.inv_step, S.q0, S.lq0_step, C.cac);
    } else {
        // Eq. (13) tail: at most 1.6 e^-x for x > 1; anything for a smaller x
        const float x = qc > S.q0 ? fmaf(C.thi_b, Ec, C.thi_a) : fmaf(C.tlo_b, Ec, C.tlo_a);
        if (!(x > 1.0f)) return __int_as_float(0x7f800000);
        stat += C.cac != 0.0f ? 1.0f : fmaf(-1.44268f, x, 0.7f + 1e-5f * x);
    }
    return kin + stat + 2.0f;
}

// FP64 words of sample group g: the four Philox words of every block.
template <int D, typename Keys>
__device__ __forceinline__ void group_words64(uint32_t* w, uint32_t g, uint32_t itn, uint32_t call, uint32_t task,
                                              const Keys& rk) {
    using S = StreamShape<D, false>;
    const uint32_t b0 = g * S::kBlocks;            // counter word 0 is the block index mod 2^32
#pragma unroll
    for (int j = 0; j < S::kBlocks; ++j) {
        uint32_t c0 = b0 + j, c1 = itn, c2 = call, c3 = task;
        philox4x32_10(c0, c1, c2, c3, rk);
        w[4 * j + 0] = c0;
        w[4 * j + 1] = c1;
        w[4 * j + 2] = c2;
        w[4 * j + 3] = c3;
    }
}

// The samples of one segment.  map32: the map table rounded to FP32; tab: the
// function tables; setup: this segment's FP64 constants, written here; all in
// shared memory.
template <int NLEG>
__device__ __forceinline__ void run_samples64(const EvalParams& P, const Segment& seg, const SideDesc& sd,
                                              const TaskDesc& td, const TaskConst& tc, const double* s_spline,
                                              const Real2<double>* s_map, const Real2<float>* s_map32,
                                              double* w_hist, const double* tab, SegSetup<double, NLEG>* s_setup,
                                              uint32_t* s_queue, Acc<double>& acc_w, Acc<double>& acc_w2) {
    constexpr int NI = NLEG - 2;
    constexpr int D = 3 * NI;
    using SS = StreamShape<D, false>;
    constexpr int G = SS::kGroup;
    const Geometry& g = P.geo;
    const int nb = td.nbins;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) {
        SegSetup<double, NLEG> st;
        seg_setup<double, NLEG>(P, sd, td, tc, &st);
        *s_setup = st;
    }
    SegSetup<float, NLEG> s32;
    seg_setup32<NLEG>(P.tconst32[seg.task], &s32);
    // what the largest weight's exponent is lowered by: the bound leaves |c0| out
    // (c0 < 0: a Fermi-Dirac gain task observed where f > 1)
    const float below = lg2_ftz(fmaxf(fabsf(static_cast<float>(tc.c0)), 1e-37f)) + kDropBits +
                        static_cast<float>(64 - __clzll(static_cast<long long>(td.neval)));
    __syncthreads();
    const SegConst<double, NLEG>& C = s_setup->C;
    const double* knots = s_spline + g.n_species * 4 * (g.n_grid - 1);
    const int ncoef = 4 * (g.n_grid - 1);
    const uint32_t call = P.ts->call, task = td.gid;
    uint32_t* q = s_queue + (tid >> 5) * (2 * D * kQueueSlots);
    const uint32_t lanes_below = (1u << lane) - 1u;
    int qn = 0;                             // queued samples (warp-uniform)
    int wmax = 0;                           // high word of the largest |w_n| evaluated by this warp
    float cutoff = -3.0e38f;                // samples with log2_weight_bound below this cannot matter

    auto drain = [&](int slot) {
        double y[D], dy[D];
        uint64_t bins[2] = {};                       // 8 bits per dimension, 6 dimensions per word
#pragma unroll
        for (int d = 0; d < D; ++d) {
            uint32_t b;
            dy[d] = map_point64(q[(2 * d) * kQueueSlots + slot], q[(2 * d + 1) * kQueueSlots + slot], nb, s_map + d * nb,
                                &y[d], &b).dy;
            bins[d / 6] |= static_cast<uint64_t>(b) << (8 * (d % 6));
        }
        bool rare;
        double w = weight64<NLEG>(C, y, dy, s_spline, knots, g, s32, s_setup->q0, s_setup->qN, ncoef, tab, &rare);
        if (rare)
            w = plain_weight64<NLEG>(q + slot, nb, s_map, s_setup, s_spline, g.n_grid, g.n_species, g.log_spaced);
        const double w2 = w * w;
        acc_w.add(w);
        acc_w2.add(w2);
        if (__double_as_longlong(w2) != 0) {
            // each lane starts at another dimension: an FP64 shared-memory
            // addition is a compare-and-swap loop, and its rounds follow the
            // number of lanes on one increment (3.1 -> about 1.3 rounds)
            int d = lane % D;
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const uint32_t b = static_cast<uint32_t>((d < 6 ? bins[0] >> (8 * d) : bins[1] >> (8 * (d - 6))) & 0xFFu);
                atomicAdd(&w_hist[d * nb + b], w2);
                d = d + 1 == D ? 0 : d + 1;
            }
        }
        return __double2hiint(w) & 0x7fffffff;
    };

    const uint32_t g1 = static_cast<uint32_t>(seg.g1), N = static_cast<uint32_t>(td.neval);
    // One sample per lane and turn; the last turn has none and empties the queue.
    // The drain stands here once: with one per sample of a group and one for the
    // rest, the loop's code was past what the SM's instruction caches hold
    // (1e5 samples x 2: 2 -> 3, 64 points 4.75 -> 3.08 ms, 2 -> 4, 64 points 5.69 ->
    // 4.72 ms; massless 2 -> 2, 128 points 9.81 -> 9.54 ms).
    uint32_t gb = static_cast<uint32_t>(seg.g0) + (tid & ~31);
    uint32_t uw[4 * SS::kBlocks];
    int sgi = 0;
    for (;;) {
        const bool more = gb < g1;
        if (more) {
            const uint32_t grp = gb + lane;
            if (G == 1 || sgi == 0) {
                group_words64<D>(uw, grp, P.itn, call, task, P.rk);
            } else {
#pragma unroll
                for (int k = 0; k < 2 * D; ++k) uw[k] = uw[(G > 1 ? 2 * D : 0) + k];
            }
            const bool valid = grp < g1 && grp * G + sgi < N;
            float y[D], jac = 1.0f;
            uint32_t frac[D], top_frac = 0;
#pragma unroll
            for (int d = 0; d < D; ++d)
                jac *= map_point32(uw[2 * d], uw[2 * d + 1], nb, s_map32 + d * nb, &y[d], &frac[d]);
#pragma unroll
            for (int d = 0; d < D; d += 2) top_frac = __vimax3_u32(top_frac, frac[d], frac[d + 1 < D ? d + 1 : d]);
            float gauss;
            const float l = log2_weight_bound<NLEG, true>(s32, P, y, jac, &gauss);
            const bool keep = valid && !(gauss < -1100.0f) && (near_edge(top_frac, nb) || !(l < cutoff));
            const uint32_t vote = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int slot = qn + __popc(vote & lanes_below);     // < 2 * 32
#pragma unroll
                for (int k = 0; k < 2 * D; ++k) q[k * kQueueSlots + slot] = uw[k];
            }
            qn += __popc(vote);
            if (++sgi == G) {
                sgi = 0;
                gb += blockDim.x;
            }
            if (qn < 32) continue;
        }
        __syncwarp();
        const int hi = lane < qn ? drain(lane) : 0;
        if (!more) break;
        const int top = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(hi)));
        if (top > wmax && top < 0x7FE00000) {
            wmax = top;
            cutoff = static_cast<float>((top >> 20) - 1023) - below;
        }
        __syncwarp();
        if (lane < qn - 32) {
#pragma unroll
            for (int k = 0; k < 2 * D; ++k) q[k * kQueueSlots + lane] = q[k * kQueueSlots + 32 + lane];
        }
        __syncwarp();
        qn -= 32;
    }
}

}  // namespace best

// FP64 kernels around the sample kernel: time state and spline construction
// (Sec. 3B) with its tangent and transpose, per-task constants, iteration reduction and VEGAS refinement,
// assembly of C_a (Eq. (7)) and the Euler / Heun updates (Sec. 3C).
#include <cmath>
#include <cstdint>

#include "internal.cuh"

namespace best {

// Scale factor a(t) (Sec. 3E).
__device__ inline double scale_factor(const Geometry& g, double t) {
    return g.expansion ? g.a0 * sqrt(t / g.t0) : 1.0;
}

// Tridiagonal solve with the factors of a SplinePlan (or its transpose), by
// one warp, in place in shared memory: y holds r_k d_k on entry.  Both
// substitutions are first-order recurrences v_k = b_k + P_k v_{k-1}: every
// lane runs its own contiguous rows from 0 while multiplying up the P_k, the
// lanes' affine maps are combined by a shuffle scan, and the rows are run
// again from the carry.  An FP64 operation of a warp takes the pipe for 64
// cycles whatever its lanes do, so the 3 n / 32 + 10 operations here replace
// 3 n dependent ones: 120 us -> 8 us for the whole spline build at n = 256.
// Rows per lane are odd so that the lanes' shared-memory rows fall in
// different banks.
__device__ inline void tri_solve_warp(int m, double* y, const double* g, const double* c) {
    const int lane = threadIdx.x & 31;
    const int q = ((m + 31) / 32) | 1;
    const int k0 = min(lane * q, m), k1 = min(k0 + q, m);
    double v = 0.0, P = 1.0;
    for (int k = k0; k < k1; ++k) {
        v = fma(-g[k], v, y[k]);
        P *= -g[k];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double vo = __shfl_up_sync(0xffffffffu, v, o), Po = __shfl_up_sync(0xffffffffu, P, o);
        if (lane >= o) {
            v = fma(P, vo, v);
            P *= Po;
        }
    }
    v = __shfl_up_sync(0xffffffffu, v, 1);
    if (lane == 0) v = 0.0;
    for (int k = k0; k < k1; ++k) {
        v = fma(-g[k], v, y[k]);
        y[k] = v;
    }
    v = 0.0;
    P = 1.0;
    for (int k = k1 - 1; k >= k0; --k) {
        v = fma(-c[k], v, y[k]);
        P *= -c[k];
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const double vo = __shfl_down_sync(0xffffffffu, v, o), Po = __shfl_down_sync(0xffffffffu, P, o);
        if (lane + o < 32) {
            v = fma(P, vo, v);
            P *= Po;
        }
    }
    v = __shfl_down_sync(0xffffffffu, v, 1);
    if (lane == 31) v = 0.0;
    for (int k = k1 - 1; k >= k0; --k) {
        v = fma(-c[k], v, y[k]);
        y[k] = v;
    }
}

// Right-hand side r_k d_k of the second-derivative system of (q_j, f_j) in
// Y[k] and the factors in G, Cp (shared memory, by every thread).
__device__ inline void notaknot_rows(const SplinePlan& pl, const double* f, double* Y, double* G, double* Cp) {
    const double* ih = pl.inv_h();
    for (int k = threadIdx.x; k < pl.n - 2; k += blockDim.x) {
        const double lo = (f[k + 1] - f[k]) * ih[k], hi = (f[k + 2] - f[k + 1]) * ih[k + 1];
        Y[k] = 6.0 * (hi - lo) * pl.r()[k];
        G[k] = pl.g()[k];
        Cp[k] = pl.c()[k];
    }
}

// Interval coefficients of the spline with second derivatives M_{k+1} = X[k].
__device__ inline void spline_coefs(const SplinePlan& pl, const double* __restrict__ knots, const double* f,
                                    const double* X, double* coef64, float* coef32) {
    const int n = pl.n;
    const double* e = pl.ends();
    auto M = [&](int j) {
        if (j == 0) return e[0] * X[0] - e[1] * X[1];
        if (j == n - 1) return e[2] * X[n - 3] - e[3] * X[n - 4];
        return X[j - 1];
    };
    for (int j = threadIdx.x; j < n - 1; j += blockDim.x) {
        const double hj = knots[j + 1] - knots[j], ih = pl.inv_h()[j];
        const double m0 = M(j), m1 = M(j + 1);
        const double c1 = (f[j + 1] - f[j]) * ih - hj * (2.0 * m0 + m1) * (1.0 / 6.0);
        const double c2 = 0.5 * m0;
        const double c3 = (m1 - m0) * ih * (1.0 / 6.0);
        reinterpret_cast<double2*>(coef64)[2 * j] = make_double2(f[j], c1);
        reinterpret_cast<double2*>(coef64)[2 * j + 1] = make_double2(c2, c3);
        reinterpret_cast<float4*>(coef32)[j] = make_float4(static_cast<float>(f[j]), static_cast<float>(c1),
                                                           static_cast<float>(c2), static_cast<float>(c3));
    }
}

__device__ inline double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Least-squares line y = a + b x through the K end points of one end of the
// grid (end 0: j < K; end 1: j >= n - K), x(j) and y(j) evaluated by one warp,
// one point per lane at a time.
template <typename X, typename Y>
__device__ inline void end_fit(int n, int K, int end, X&& x, Y&& y, double* a0, double* b) {
    const int lane = threadIdx.x & 31;
    const int j0 = end == 0 ? 0 : n - K;
    double xm = 0.0, ym = 0.0, x0 = 0.0, y0 = 0.0;
    for (int k = lane; k < K; k += 32) {
        const double xv = x(j0 + k), yv = y(j0 + k);
        if (k == lane) {
            x0 = xv;
            y0 = yv;
        }
        xm += xv;
        ym += yv;
    }
    xm = warp_sum(xm) / K;
    ym = warp_sum(ym) / K;
    double sxy = 0.0, sxx = 0.0;
    for (int k = lane; k < K; k += 32) {
        const double xc = (k == lane ? x0 : x(j0 + k)) - xm, yv = k == lane ? y0 : y(j0 + k);
        sxy += xc * (yv - ym);
        sxx += xc * xc;
    }
    *b = warp_sum(sxy) / warp_sum(sxx);
    *a0 = ym - *b * xm;
}

// ---------------------------------------------------------------------------
// First kernel of a sweep, one CTA of 256 threads per species: the time state
// (a(t), Sec. 3E; m_s(t), Sec. 3A), cleared chunk counters, and the spline of
// the species: not-a-knot cubic spline of (q_j, f_j) from the second
// derivatives M_j, and the least-squares end fits of log(1/f + eta) against
// E(q/a) (Eq. (13)).  While one warp substitutes, two others make the end fits
// and a fourth the time state.
// src_mode 0: f given; 1: f = exp(src) (log f).
// Dynamic shared memory: 4 n doubles.
// ---------------------------------------------------------------------------
__global__ void spline_build_kernel(Geometry g, SweepStart ss, const double* __restrict__ src, int src_mode,
                                    const double* __restrict__ knots, SplinePlan pl, TimeState* ts,
                                    SpeciesConst* sc, double* fgrid, double* coef64,
                                    float* coef32) {
    extern __shared__ double sh[];
    const int n = g.n_grid;
    const int s = blockIdx.x;
    double* f = sh;
    double* Y = sh + n;
    double* G = sh + 2 * n;
    double* Cp = sh + 3 * n;
    if (blockIdx.x == 0)
        for (int k = threadIdx.x; k < ss.n_ctr; k += blockDim.x) ss.ctr[k] = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double v = src[static_cast<int64_t>(s) * n + j];
        if (src_mode == 1) v = exp(v);
        if (!(v > 0.0) || !isfinite(v)) ts->error = BEST_ERR_NUMERIC;
        f[j] = v;
        fgrid[static_cast<int64_t>(s) * n + j] = v;
    }
    __syncthreads();
    notaknot_rows(pl, f, Y, G, Cp);
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        tri_solve_warp(n - 2, Y, G, Cp);
    } else if (warp <= 3) {
        double t = ss.t_host, a, mass;
        if (ss.law) {
            if (ss.mode == 1) t = *ss.t_dev;
            if (ss.mode == 2) t = *ss.t_dev + ts->dt;
            a = scale_factor(g, t);
            mass = mass_at(ss.law[s], t);
        } else {
            a = ts->a;
            mass = ts->mass[s];
        }
        if (warp < 3) {
            const double eta = sc[s].eta;
            auto x = [&](int j) {
                const double p = knots[j] / a;
                return sqrt(p * p + mass * mass);
            };
            auto y = [&](int j) { return log(1.0 / f[j] + eta); };
            double a0, b;
            end_fit(n, g.tail_points, warp - 1, x, y, &a0, &b);
            if ((threadIdx.x & 31) == 0) {
                if (warp == 1) { sc[s].tail_lo_a = a0; sc[s].tail_lo_b = b; }
                else { sc[s].tail_hi_a = a0; sc[s].tail_hi_b = b; }
            }
        } else if (ss.law && threadIdx.x == 96) {
            ts->mass[s] = mass;
            if (s == 0) {
                ts->t = t;
                ts->a = a;
                ts->inv_a = 1.0 / a;
                if (!(a > 0.0) || !isfinite(a)) ts->error = BEST_ERR_NUMERIC;
            }
        }
    }
    __syncthreads();
    const int64_t o = static_cast<int64_t>(s) * (n - 1) * 4;
    spline_coefs(pl, knots, f, Y, coef64 + o, coef32 + o);
}

// ---------------------------------------------------------------------------
// Tangent of the spline construction in the direction u (one species per
// CTA): the interval coefficients are linear in f, so the tangent spline is
// the spline of u (no clamping); the end fits y = log(1/f + eta) = a + b E
// move by da, db from dy_j = -u_j / (f_j (1 + eta f_j)).  Also clears the
// tangent kernel's chunk counter.  256 threads; dynamic shared memory: 4 n
// doubles.
// ---------------------------------------------------------------------------
__global__ void spline_tangent_kernel(Geometry g, const double* __restrict__ u, const double* __restrict__ knots,
                                      SplinePlan pl, const double* __restrict__ fgrid,
                                      const SpeciesConst* __restrict__ sc, const TimeState* ts, int32_t* ctr,
                                      double* dcoef64, float* dcoef32, double* dtail) {
    extern __shared__ double sh[];
    const int n = g.n_grid;
    const int s = blockIdx.x;
    double* du = sh;
    double* Y = sh + n;
    double* G = sh + 2 * n;
    double* Cp = sh + 3 * n;
    if (blockIdx.x == 0 && threadIdx.x == 0) *ctr = 0;
    for (int j = threadIdx.x; j < n; j += blockDim.x) du[j] = u[static_cast<int64_t>(s) * n + j];
    __syncthreads();
    notaknot_rows(pl, du, Y, G, Cp);
    __syncthreads();
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        tri_solve_warp(n - 2, Y, G, Cp);
    } else if (warp <= 2) {
        const double eta = sc[s].eta, mass = ts->mass[s], a = ts->a;
        const double* f = fgrid + static_cast<int64_t>(s) * n;
        auto x = [&](int j) {
            const double p = knots[j] / a;
            return sqrt(p * p + mass * mass);
        };
        auto y = [&](int j) { return -du[j] / (f[j] * (1.0 + eta * f[j])); };
        double da, db;
        end_fit(n, g.tail_points, warp - 1, x, y, &da, &db);
        if ((threadIdx.x & 31) == 0) {
            dtail[s * 4 + 2 * (warp - 1)] = da;
            dtail[s * 4 + 2 * (warp - 1) + 1] = db;
        }
    }
    __syncthreads();
    const int64_t o = static_cast<int64_t>(s) * (n - 1) * 4;
    spline_coefs(pl, knots, du, Y, dcoef64 + o, dcoef32 + o);
}

// ---------------------------------------------------------------------------
// Transpose of the spline construction for one species per CTA (256 threads):
// the interval coefficients are linear in f through the second derivatives M
// (not-a-knot tridiagonal system), so df = L^T dcoef; plus the tail fits'
// dependence on the end values f_j and, through E(q_j/a), on the mass.  Every
// row is a gather over its neighbours, the transposed system is solved like
// the forward one (one thread walking the rows took 980 us at n = 256).
// Dynamic shared memory: 4 n doubles.
// ---------------------------------------------------------------------------
__global__ void spline_adjoint_kernel(Geometry g, const double* __restrict__ knots, SplinePlan pl,
                                      const double* __restrict__ fgrid, const SpeciesConst* __restrict__ sconst,
                                      const TimeState* ts, const double* __restrict__ gcoef,
                                      const double* __restrict__ gtail, double* gf, double* gm) {
    extern __shared__ double sh[];
    const int n = g.n_grid, m = n - 2;
    const int s = blockIdx.x;
    double* gM = sh;                   // dL/dM_j
    double* Y = sh + n;
    double* G = sh + 2 * n;
    double* Cp = sh + 3 * n;
    const double* gc = gcoef + static_cast<int64_t>(s) * (n - 1) * 4;
    const double* f = fgrid + static_cast<int64_t>(s) * n;
    const double* ih = pl.inv_h();
    double* out = gf + static_cast<int64_t>(s) * n;
    // interval j: c1 = (f_{j+1} - f_j)/h - h (2 M_j + M_{j+1})/6, c2 = M_j/2, c3 = (M_{j+1} - M_j)/(6 h)
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double v = 0.0;
        if (j < n - 1) {
            const double hj = knots[j + 1] - knots[j];
            v += -gc[4 * j + 1] * hj * (1.0 / 3.0) + 0.5 * gc[4 * j + 2] - gc[4 * j + 3] * ih[j] * (1.0 / 6.0);
        }
        if (j > 0) {
            const double hp = knots[j] - knots[j - 1];
            v += -gc[4 * (j - 1) + 1] * hp * (1.0 / 6.0) + gc[4 * (j - 1) + 3] * ih[j - 1] * (1.0 / 6.0);
        }
        gM[j] = v;
    }
    __syncthreads();
    // the end derivatives M_0 and M_{n-1} in terms of M_1, M_2 and M_{n-2}, M_{n-3} (the same
    // rows when n = 4)
    if (threadIdx.x == 0) {
        const double* e = pl.ends();
        gM[1] += e[0] * gM[0];
        gM[2] -= e[1] * gM[0];
        gM[n - 2] += e[2] * gM[n - 1];
        gM[n - 3] -= e[3] * gM[n - 1];
    }
    __syncthreads();
    for (int k = threadIdx.x; k < m; k += blockDim.x) {
        Y[k] = gM[k + 1] * pl.r()[k];
        G[k] = pl.gT()[k];
        Cp[k] = pl.cT()[k];
        gM[k + 1] = 0.0;                  // from here on the low end's tail terms
    }
    if (threadIdx.x < 2) gM[threadIdx.x * (n - 1)] = 0.0;
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __shared__ double mass_grad[2];
    if (warp == 0) {
        tri_solve_warp(m, Y, G, Cp);
    } else if (warp <= 2) {
        // tail fits (least squares of y = log(1/f + eta) against x = E(q/a)):
        // the low end's terms go to gM[0, K), the high end's to out[n - K, n)
        const int end = warp - 1, K = g.tail_points, j0 = end == 0 ? 0 : n - K;
        const double ga = gtail[s * 4 + 2 * end], gb = gtail[s * 4 + 2 * end + 1];
        const double eta = sconst[s].eta, mass = ts->mass[s], aa = ts->a;
        double dm = 0.0;
        if (ga != 0.0 || gb != 0.0) {
            auto x = [&](int j) {
                const double p = knots[j] / aa;
                return sqrt(p * p + mass * mass);
            };
            double xm = 0.0, ym = 0.0;
            for (int k = lane; k < K; k += 32) {
                xm += x(j0 + k);
                ym += log(1.0 / f[j0 + k] + eta);
            }
            xm = warp_sum(xm) / K;
            ym = warp_sum(ym) / K;
            double sxx = 0.0, sxy = 0.0;
            for (int k = lane; k < K; k += 32) {
                const double xc = x(j0 + k) - xm;
                sxx += xc * xc;
                sxy += xc * (log(1.0 / f[j0 + k] + eta) - ym);
            }
            sxx = warp_sum(sxx);
            sxy = warp_sum(sxy);
            const double b = sxy / sxx;
            for (int k = lane; k < K; k += 32) {
                const int j = j0 + k;
                const double xv = x(j), yv = log(1.0 / f[j] + eta);
                const double dady = 1.0 / K - xm * (xv - xm) / sxx;
                const double dbdy = (xv - xm) / sxx;
                const double dydf = -1.0 / (f[j] * (1.0 + eta * f[j]));
                const double df = (ga * dady + gb * dbdy) * dydf;
                if (end == 0) gM[j] = df;
                else out[j] += df;
                const double dbdx = ((yv - ym) - 2.0 * b * (xv - xm)) / sxx;
                const double dadx = -b / K - xm * dbdx;
                if (xv > 0.0) dm += (ga * dadx + gb * dbdx) * mass / xv;
            }
        }
        dm = warp_sum(dm);
        if (lane == 0) mass_grad[end] = dm;
    }
    __syncthreads();
    if (threadIdx.x == 0) gm[s] += mass_grad[0] + mass_grad[1];
    // d_k = 6 ((f_{k+2} - f_{k+1})/h_{k+1} - (f_{k+1} - f_k)/h_k) and the slope terms of c0, c1
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        double v = out[j] + gM[j];
        if (j < n - 1) v += gc[4 * j] - gc[4 * j + 1] * ih[j];
        if (j > 0) v += gc[4 * (j - 1) + 1] * ih[j - 1];
        if (j < m) v += 6.0 * Y[j] * ih[j];                                    // f_j in row k = j
        if (j >= 1 && j - 1 < m) v -= 6.0 * Y[j - 1] * (ih[j] + ih[j - 1]);    // k = j - 1
        if (j >= 2) v += 6.0 * Y[j - 2] * ih[j - 1];                           // k = j - 2
        out[j] = v;
    }
}

// ---------------------------------------------------------------------------
// Per-task constants of the sweep and reset of the iteration accumulators.
// ---------------------------------------------------------------------------
// Accumulation scale: the kernel sums w_n = w / (K scale).  With a previous
// estimate I of the task (last sweep) scale = |I| / K, so that w_n averages
// to about 1; otherwise scale = f_obs.  The scale is kept within 2^+-100 of
// the observed-leg factor so that obs_factor / scale fits in FP32.
__device__ inline double clamp_scale(double scale, double obs_factor) {
    if (!(obs_factor > 0.0)) return scale > 0.0 && isfinite(scale) ? scale : 1.0;
    const double lo = obs_factor * 7.888609052210118e-31, hi = obs_factor * 1.2676506002282294e30;
    if (!(scale > 0.0) || !isfinite(scale)) return obs_factor;
    return scale < lo ? lo : (scale > hi ? hi : scale);
}

// One thread per task; FP64 operations take an SM partition's pipe for 64
// cycles per warp, so the CTAs are single warps (spread over the SMs), what
// depends on neither time nor distribution comes from SideConst, and the
// common a = 1 skips its powers (13.7 -> 6.9 us for 512 tasks).
__global__ void prepare_kernel(Geometry g, const SideDesc* __restrict__ sides,
                               const TaskDesc* __restrict__ tasks, const double* __restrict__ knots,
                               const double* __restrict__ fgrid, const TimeState* ts,
                               const double* __restrict__ prev, TaskConst* tconst, TaskAcc* acc, int reset_acc,
                               const double* __restrict__ width, const SpeciesConst* __restrict__ sconst,
                               SegConst32* tconst32, const SideConst* __restrict__ sideconst) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.n_tasks) return;
    const TaskDesc td = tasks[t];
    const SideDesc& sd = sides[td.si];
    const SideConst kc = sideconst[td.si];
    const double a = ts->a;
    const double m = ts->mass[sd.species_obs];
    double p = knots[td.point], a3 = 1.0;               // a^{-3(n-2)}
    if (a != 1.0) {
        p /= a;
        const double ia = ts->inv_a, ia3 = ia * ia * ia;
        for (int k = 2; k < sd.n; ++k) a3 *= ia3;
    }
    const double E = sqrt(p * p + m * m);
    TaskConst c;
    c.p_obs = p;
    c.E_obs = E;
    c.f_obs = fgrid[static_cast<int64_t>(sd.species_obs) * g.n_grid + td.point];
    // fractional width (App. C): the per-sample factor sigma_ref / sigma with
    // sigma_ref = w E_obs is applied in the sample kernel
    c.wfrac = sd.width_mode == 0 ? 0.0 : (width ? width[sd.process] : sd.width0);
    c.inv_E_obs = 1.0 / E;
    c.K = kc.kfac * a3 * c.inv_E_obs;
    if (sd.width_mode != 0) c.K = c.K * c.inv_E_obs / c.wfrac;
    c.obs_factor = td.term == 1 ? c.f_obs : 1.0 + sd.eta_obs * c.f_obs;
    const double est = prev[t];
    c.scale = clamp_scale(est > 0.0 && c.K > 0.0 ? est / c.K : (c.f_obs > 0.0 ? c.f_obs : 1.0), c.obs_factor);
    // the observed leg's own cut (App. A) removes the whole task
    c.c0 = E < g.e_cut ? 0.0 : c.obs_factor / c.scale;
    c.gauss_k = c.wfrac > 0.0 ? -2.0 * 1.4426950408889634 / (c.wfrac * c.wfrac) : kc.gauss_k;
    c.inv_sig2_abs = kc.inv_sig2;
    c.four_over_w2 = c.wfrac > 0.0 ? 4.0 / (c.wfrac * c.wfrac) : 0.0;
    tconst[t] = c;
    if (tconst32) tconst32[t] = seg_const32(sd, td, c, *ts, sconst, g);
    if (!reset_acc) return;
    TaskAcc z;
    z.sum_inv_var = 0.0; z.sum_mean_inv_var = 0.0; z.sum_exact = 0.0; z.n_exact = 0.0;
    z.mean = 0.0; z.err = 0.0;
    acc[t] = z;
}

// ---------------------------------------------------------------------------
// Adaptive stratified sampling (VEGAS+): per-task hypercube allocation m_h
// (items of kItem samples, at least one per hypercube) and the hypercube of
// every item, items in hypercube order.  One CTA of 256 threads per task.
// ---------------------------------------------------------------------------
namespace {

// Exclusive prefix of v over the CTA (v of thread k at position k), with the
// CTA total in *total; s: 256 int64 of shared memory.
__device__ int64_t cta_exclusive_scan(int64_t v, int64_t* s, int64_t* total) {
    s[threadIdx.x] = v;
    __syncthreads();
    for (int o = 1; o < static_cast<int>(blockDim.x); o <<= 1) {
        const int64_t a = static_cast<int>(threadIdx.x) >= o ? s[threadIdx.x - o] : 0;
        __syncthreads();
        s[threadIdx.x] += a;
        __syncthreads();
    }
    const int64_t incl = s[threadIdx.x];
    *total = s[blockDim.x - 1];
    __syncthreads();
    return incl - v;
}

// f(h, first, count, scope) for every hypercube h of a task, first and count
// its items (m, in hypercube order).  Who calls it follows the count, so that
// neither many small hypercubes nor one that drew most of the items leaves the
// CTA idle: below 32 items one thread (scope 1), below 1024 or J / 16 (J: the
// task's items) one warp (scope 32, every lane with the same arguments), else
// every thread of the CTA (scope blockDim, together).  The caller's index within
// the scope is threadIdx.x % scope.  The items named lie in [0, J) whatever m
// holds (a loaded state's allocation is not checked): negative counts and what
// goes past J are cut off.  s, off, cnt: 256 entries of shared memory each.
template <typename F>
__device__ void for_hypercubes(const int32_t* m, int H, int64_t J, int64_t* s, int64_t* off, int32_t* cnt, F&& f) {
    const int64_t large = max(int64_t(1024), J / 16);
    int64_t base = 0;
    for (int c0 = 0; c0 < H; c0 += blockDim.x) {
        const int h = c0 + static_cast<int>(threadIdx.x);
        const int32_t m_h = h < H ? max(m[h], 0) : 0;
        int64_t tot;
        const int64_t ex = base + cta_exclusive_scan(m_h, s, &tot);
        const int32_t v = static_cast<int32_t>(min(static_cast<int64_t>(m_h), max(int64_t(0), J - ex)));
        off[threadIdx.x] = ex;
        cnt[threadIdx.x] = v;
        __syncthreads();
        if (h < H && v < 32) f(h, ex, v, 1);
        __syncwarp();
        const int nh = min(H - c0, static_cast<int>(blockDim.x));
        for (int k = threadIdx.x >> 5; k < nh; k += blockDim.x >> 5)
            if (cnt[k] >= 32 && cnt[k] < large) f(c0 + k, off[k], cnt[k], 32);
        for (int k = 0; k < nh; ++k)
            if (cnt[k] >= large) f(c0 + k, off[k], cnt[k], static_cast<int>(blockDim.x));
        base += tot;
        __syncthreads();
    }
}

__device__ void strat_write_items(const int32_t* m, int H, int64_t J, uint32_t* item_h, int64_t* s, int64_t* off,
                                  int32_t* cnt) {
    for_hypercubes(m, H, J, s, off, cnt, [&](int h, int64_t first, int32_t count, int scope) {
        for (int k = threadIdx.x % scope; k < count; k += scope)
            item_h[first + k] = static_cast<uint32_t>(h);
    });
}

__device__ void uniform_allocation(int32_t* m, int H, int64_t J) {
    for (int h = threadIdx.x; h < H; h += blockDim.x)
        m[h] = static_cast<int32_t>(J / H + (h < J % H ? 1 : 0));
}

}  // namespace

// uniform != 0: first (uniform) allocation; otherwise only the items are
// rebuilt from the stored allocation (after a state load).
__global__ void strat_init_kernel(const TaskDesc* __restrict__ tasks, int32_t* strat_m, uint32_t* item_h,
                                  int uniform) {
    __shared__ int64_t s[256], off[256];
    __shared__ int32_t cnt[256];
    const TaskDesc td = tasks[blockIdx.x];
    if (td.strat_H == 0) return;
    int32_t* m = strat_m + td.strat_off_h;
    if (uniform) {
        uniform_allocation(m, td.strat_H, td.strat_J);
        __syncthreads();
    }
    strat_write_items(m, td.strat_H, td.strat_J, item_h + td.strat_off_item, s, off, cnt);
}

// After the sample kernel of an iteration, one CTA per active task: per
// hypercube S1 = sum w, S2 = sum w^2 from its items (fixed order), the
// iteration estimate I = (1/H) sum_h S1_h / n_h and variance
// (1/H^2) sum_h s_h^2 / n_h (n_h = kItem m_h), written to est[4 t ..] with an
// underflow flag (S2 < S1^2 / n violated, i.e. FP32 squares underflowed, in
// hypercubes holding more than 1e-6 of sum_h |S1_h| / n_h); then the
// next allocation m_h = 1 + floor((J - H) d_h / sum d), d_h = (s_h^2)^(beta/2),
// the remaining items one each to h = 0, 1, ... (uniform if every d_h = 0 or one
// is infinite),
// and the items rebuilt.  An underflowed iteration keeps its allocation.
__global__ void __launch_bounds__(256, 4) strat_refine_kernel(const TaskDesc* __restrict__ tasks, const int32_t* __restrict__ active,
                                    const double* __restrict__ item_rec, int32_t* strat_m, double* strat_d,
                                    double* strat_s2, uint32_t* item_h, double* est) {
    __shared__ int64_t s[256], off[256];
    __shared__ int32_t cnt[256];
    __shared__ double r0[256], r1[256], r2[256], r3[256], r4[256];
    __shared__ int64_t si[256];
    const int t = active[blockIdx.x];
    const TaskDesc td = tasks[t];
    if (td.strat_H == 0) return;
    const int H = td.strat_H;
    const int64_t J = td.strat_J;
    int32_t* m = strat_m + td.strat_off_h;
    double* S1h = strat_d + td.strat_off_h;      // sum w per hypercube, then d_h
    double* S2h = strat_s2 + td.strat_off_h;
    const double2* rec = reinterpret_cast<const double2*>(item_rec) + td.strat_off_item;
    // per-hypercube sums of its items' records, in an order fixed by the
    // allocation: coalesced loads, two FP64 additions per record and thread, one
    // chain of additions per warp (lower lanes w, upper lanes w^2).  (Per-thread
    // runs of items whose ends one thread added up took 204 us for 512 tasks of
    // 12500 items, most of it that thread; now 97 us, and 437 us for 125000 items
    // (523).  The additions alone take the FP64 pipe 22 and 220 us.)
    __shared__ double s_w[16];
    for_hypercubes(m, H, J, s, off, cnt, [&](int h, int64_t first, int32_t count, int scope) {
        double s1 = 0.0, s2 = 0.0;
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const double2* p = rec + first;
        int k = threadIdx.x % scope;
        if (k + 3 * scope < count) {
            // four records in flight while the four before are added
            double2 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = p[k + u * scope];
            k += 4 * scope;
            for (; k + 3 * scope < count; k += 4 * scope) {
                double2 y[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) y[u] = p[k + u * scope];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    s1 += x[u].x;
                    s2 += x[u].y;
                    x[u] = y[u];
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                s1 += x[u].x;
                s2 += x[u].y;
            }
        }
        for (; k < count; k += 4 * scope) {
            double2 x[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) x[u] = k + u * scope < count ? p[k + u * scope] : make_double2(0.0, 0.0);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                if (k + u * scope < count) {
                    s1 += x[u].x;
                    s2 += x[u].y;
                }
        }
        if (scope == 1) {
            S1h[h] = s1;
            S2h[h] = s2;
            return;
        }
        const bool up = lane >= 16;
        double v = up ? s2 : s1;
        v += __shfl_xor_sync(0xffffffffu, up ? s1 : s2, 16);
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        double* S = up ? S2h : S1h;
        if (scope == 32) {
            if ((lane & 15) == 0) S[h] = v;
            return;
        }
        if ((lane & 15) == 0) s_w[2 * warp + (up ? 1 : 0)] = v;
        __syncthreads();
        if (warp == 0 && (lane & 15) == 0) {
            double sum = 0.0;
            for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) sum += s_w[2 * w + (up ? 1 : 0)];
            S[h] = sum;
        }
        __syncthreads();
    });
    __syncthreads();
    double a_mean = 0.0, a_var = 0.0, a_d = 0.0, a_abs = 0.0, a_bad = 0.0;
    for (int h = threadIdx.x; h < H; h += blockDim.x) {
        const double S1 = S1h[h], S2 = S2h[h];
        const double n = static_cast<double>(kItem) * static_cast<double>(m[h]);
        const double q = S1 * S1 / n;
        double s2v = (S2 - q) / (n - 1.0);
        s2v = s2v > 0.0 ? s2v : 0.0;
        if (S2 < (1.0 - 1e-6) * q) a_bad += fabs(S1) / n;
        a_abs += fabs(S1) / n;
        a_mean += S1 / n;
        a_var += s2v / n;
        const double d = pow(s2v, 0.5 * td.strat_beta);
        S1h[h] = d;
        a_d += d;
    }
    r0[threadIdx.x] = a_mean;
    r1[threadIdx.x] = a_var;
    r2[threadIdx.x] = a_d;
    r3[threadIdx.x] = a_abs;
    r4[threadIdx.x] = a_bad;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (static_cast<int>(threadIdx.x) < o) {
            r0[threadIdx.x] += r0[threadIdx.x + o];
            r1[threadIdx.x] += r1[threadIdx.x + o];
            r2[threadIdx.x] += r2[threadIdx.x + o];
            r3[threadIdx.x] += r3[threadIdx.x + o];
            r4[threadIdx.x] += r4[threadIdx.x + o];
        }
        __syncthreads();
    }
    const double sum_d = r2[0];
    // underflowed hypercubes (FP32 squares of weights near the end of the
    // range) matter only when they carry a noticeable part of the estimate
    const bool underflow = r4[0] > 1e-6 * r3[0];
    if (threadIdx.x == 0) {
        est[4 * t] = r0[0] / H;
        est[4 * t + 1] = r1[0] / (static_cast<double>(H) * H);
        est[4 * t + 2] = underflow ? 1.0 : 0.0;
    }
    if (underflow) return;
    __syncthreads();
    // (an infinite sum -- FP32 squares that overflowed -- has no shares: inf / inf would become the integer
    // of a NaN, -2^31)
    if (sum_d > 0.0 && isfinite(sum_d)) {
        int64_t cnt = 0;
        for (int h = threadIdx.x; h < H; h += blockDim.x) {
            const int32_t v = 1 + static_cast<int32_t>(floor(static_cast<double>(J - H) * S1h[h] / sum_d));
            m[h] = v;
            cnt += v;
        }
        si[threadIdx.x] = cnt;
        __syncthreads();
        for (int o = blockDim.x / 2; o > 0; o >>= 1) {
            if (static_cast<int>(threadIdx.x) < o) si[threadIdx.x] += si[threadIdx.x + o];
            __syncthreads();
        }
        const int64_t rest = J - si[0];
        __syncthreads();
        if (rest >= 0) {
            for (int h = threadIdx.x; h < H; h += blockDim.x)
                if (h < rest) m[h] += 1;
        } else {
            uniform_allocation(m, H, J);      // rounding overshoot (never seen): start afresh
        }
    } else {
        uniform_allocation(m, H, J);
    }
    __syncthreads();
    strat_write_items(m, H, J, item_h + td.strat_off_item, s, off, cnt);
}

// ---------------------------------------------------------------------------
// End of one VEGAS iteration, one CTA per active task and integrated leg (its
// three dimensions): sum the task's segment records in a fixed order
// (deterministic), form the iteration estimate and its variance, add them to
// the combination accumulators, and refine the map (Lepage): smooth the
// per-increment sums of w^2 with the (7,1)/8, (1,6,1)/8, (1,7)/8 stencil,
// normalise, compress with ((1-d)/ln(1/d))^alpha, and re-partition into equal
// shares of the compressed weight.  A normalised share below 1e-30 counts as an
// empty increment (weight 0, like an exact zero) so that the map does not
// depend on where underflow of w^2 falls.
//
// Bound by the FP64 pipe (64 cycles per warp operation) and by dependent
// loads: one warp per dimension runs its dimension from smoothing to edges
// without block barriers (warp-wide sums and scans, comparisons as integers),
// while a fourth warp makes the task's scalars; the legs' CTAs spread a small
// problem over the SMs.  FP32 2 -> 2: 17.8 -> 8.7 us for 64 tasks, 83 -> 52 us for
// 512; 486 -> 302 us for 6144 tasks of 2 -> 2 and 2 -> 3.  Dynamic shared memory: refine_doubles(nbins_max) doubles.
// ---------------------------------------------------------------------------
__global__ void refine_kernel(Geometry g, const SideDesc* __restrict__ sides,
                              const TaskDesc* __restrict__ tasks, const TaskConst* tconst,
                              const int32_t* __restrict__ active, const int32_t* __restrict__ task_seg,
                              const Segment* __restrict__ segs, const double* __restrict__ partials,
                              double* edges, TaskAcc* acc, TaskConst* tconst_next,
                              const double* __restrict__ strat_est, SegConst32* tconst32, float2* map32, int legs) {
    extern __shared__ double hist[];
    __shared__ int s_underflow;
    const int a = blockIdx.x / legs, leg = blockIdx.x - a * legs;
    const int t = active[a];
    const int s0 = task_seg[a], s1 = task_seg[a + 1];
    const TaskDesc& td = tasks[t];
    const int nb = td.nbins;
    if (3 * leg >= td.dim) return;
    const int E = 3 * nb;
    double* head = hist + E;                   // sum w, sum w^2
    double* sm = head + 2;                     // smoothed, then compressed weights [3][nb]
    double* olde = sm + E;                     // old edges [3][nb + 1]
    double* rom = olde + E + 3;                // reciprocals of the compressed weights [3][nb]
    double* cum = rom + E;                     // running sums of the compressed weights [3][nb + 1]
    double* e_task = edges + static_cast<int64_t>(t) * g.map_stride + 3 * leg * (nb + 1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double old0 = tid < E + 3 ? e_task[tid] : 0.0;           // (under way with the records)
    {
        // the records in segment order (one after the other in memory); eight loads in flight at a time
        const int64_t rec = record_doubles(td.dim, nb);
        const double* part = partials + segs[s0].part;
        const int n = s1 - s0;
        for (int k = tid; k < E + 2; k += blockDim.x) {
            const double* p = part + (k < E ? 2 + leg * E + k : k - E);
            double v = 0.0;
            int s = 0;
            for (; s + 8 <= n; s += 8, p += 8 * rec) {
                double x[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) x[u] = p[u * rec];
#pragma unroll
                for (int u = 0; u < 8; ++u) v += x[u];
            }
            for (; s < n; ++s, p += rec) v += *p;
            hist[k] = v;
        }
    }
    if (tid < E + 3) olde[tid] = old0;
    for (int k = tid + blockDim.x; k < E + 3; k += blockDim.x) olde[k] = e_task[k];
    __syncthreads();
    if (warp > 3) return;
    if (warp == 3) {
        // Sum w^2 >= (sum w)^2 / N holds exactly; if the computed sums violate
        // it, squares of tiny weights underflowed (FP32 path with a poor scale):
        // the iteration is discarded (no estimate, no refinement) and only the
        // scale is corrected for the next iteration.
        const double N = static_cast<double>(td.neval);
        double mean_n, var_n;
        bool underflow;
        if (td.strat_H > 0) {
            // stratified: estimate, variance and underflow flag from strat_refine_kernel
            mean_n = strat_est[4 * t];
            var_n = strat_est[4 * t + 1];
            underflow = strat_est[4 * t + 2] != 0.0;
        } else {
            mean_n = head[0] / N;
            const double sq = head[1] / N;
            underflow = sq < (1.0 - 1e-6) * mean_n * mean_n;
            var_n = N > 1.0 ? (sq - mean_n * mean_n) / (N - 1.0) : 0.0;
            var_n = var_n > 0.0 ? var_n : 0.0;
        }
        if (lane == 0) s_underflow = underflow ? 1 : 0;
        __syncwarp();
        asm volatile("bar.arrive 1, 128;" ::: "memory");
        if (leg != 0 || lane != 0) return;
        const TaskConst& c = tconst[t];
        const double K = c.K, old_scale = c.scale, obs_factor = c.obs_factor, c0 = c.c0;
        const double sc = K * old_scale;
        const double mean = mean_n * sc;
        const double var = var_n * sc * sc;
        if (!underflow) {
            TaskAcc& A = acc[t];
            if (var > 0.0) {
                A.sum_inv_var += 1.0 / var;
                A.sum_mean_inv_var += mean / var;
            } else {
                A.sum_exact += mean;
                A.n_exact += 1.0;
            }
        }
        if (mean_n != 0.0) {
            const double scale = clamp_scale(fabs(mean_n) * old_scale, obs_factor);
            const double next = c0 == 0.0 ? 0.0 : obs_factor / scale;   // a cut observed leg stays cut
            tconst_next[t].scale = scale;
            tconst_next[t].c0 = next;
            if (tconst32) tconst32[t].c0 = static_cast<float>(next);
        }
        return;
    }
    // ---- one dimension per warp ----
    const bool f32 = g.precision == BEST_FP32;
    const double* dd = hist + warp * nb;
    sm += warp * nb;
    rom += warp * nb;
    cum += warp * (nb + 1);
    olde += warp * (nb + 1);
    double tot = 0.0;
    for (int b = lane; b < nb; b += 32) {
        double v;
        if (b == 0) v = (7.0 * dd[0] + dd[1]) / 8.0;
        else if (b == nb - 1) v = (dd[nb - 2] + 7.0 * dd[nb - 1]) / 8.0;
        else v = (dd[b - 1] + 6.0 * dd[b] + dd[b + 1]) / 8.0;
        sm[b] = v;
        tot += v;
    }
    tot = warp_sum(tot);
    const bool refined = tot > 0.0;            // else no training data: the map is kept
    if (refined) {
        // FP32 path: the total is a sum of FP32 training data, so its
        // reciprocal is finite (an FP64 total can be subnormal)
        const double inv = f32 ? 1.0 / tot : 0.0;
        for (int b = lane; b < nb; b += 32) {
            double o, r;
            if (f32) {
                // the FP32 path's training data carry FP32 rounding: its
                // compression and reciprocal are evaluated in FP32 (FP64
                // division, log and pow run at a small fraction of the FP32
                // rate on this GPU)
                const float vf = static_cast<float>(sm[b] * inv);
                float of = 1.0f;               // v >= 1, or not a number (FP32 training data overflowed)
                if (vf < 1e-30f) of = 0.0f;    // numerically empty increment
                else if (vf < 1.0f) of = powf((1.0f - vf) / -logf(vf), static_cast<float>(td.alpha));
                o = of;
                r = of > 0.0f ? __frcp_rn(of) : 0.0f;
            } else {
                const double v = sm[b] / tot;
                if (v < 1e-30) o = 0.0;        // numerically empty increment
                else if (v >= 1.0) o = 1.0;
                else {
                    const double x = (1.0 - v) / -log(v);
                    o = td.alpha == 0.5 ? sqrt(x) : pow(x, td.alpha);
                }
                // the interpolation below multiplies by these reciprocals (o is
                // 0 or at least (1 / ln 1e30)^alpha)
                r = o > 0.0 ? 1.0 / o : 0.0;
            }
            sm[b] = o;
            rom[b] = r;
        }
        __syncwarp();
        // running sums: every lane its own increments, then a scan of the lanes
        const int per = (nb + 31) / 32, b0 = min(lane * per, nb), b1 = min(b0 + per, nb);
        double mine = 0.0;
        for (int b = b0; b < b1; ++b) mine += sm[b];
        double run = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double x = __shfl_up_sync(0xffffffffu, run, o);
            if (lane >= o) run += x;
        }
        run = __shfl_up_sync(0xffffffffu, run, 1);
        if (lane == 0) {
            run = 0.0;
            cum[0] = 0.0;
        }
        for (int b = b0; b < b1; ++b) {
            run += sm[b];
            cum[b + 1] = run;
        }
        __syncwarp();
    }
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (s_underflow) return;
    // new edge k: starting from increment 0, step to the next increment while
    // the running sum after it stays below the goal k T / nb (and an increment
    // is left): the number of j in [1, nb - 1] with cum[j] < goal, and the
    // linear interpolation inside it.  The sums and goals are not negative, so
    // they compare as integers.
    double* e = e_task + warp * (nb + 1);
    if (refined) {
        const double target = cum[nb] / nb;
        for (int k = lane; k < nb; k += 32) {
            double v = 0.0;
            if (k > 0) {
                const double goal = k * target;
                const long long gi = __double_as_longlong(goal);
                int lo = 0, hi = nb - 1;                     // first i in [0, nb - 1] with !(cum[i + 1] < goal), else nb - 1
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (__double_as_longlong(cum[mid + 1]) < gi) lo = mid + 1;
                    else hi = mid;
                }
                double fr = (goal - cum[lo]) * rom[lo];
                fr = fr < 0.0 ? 0.0 : (fr > 1.0 ? 1.0 : fr);
                v = olde[lo] + fr * (olde[lo + 1] - olde[lo]);
            }
            e[k] = v;
            sm[k] = v;                                       // (the compressed weights are done with)
        }
        if (lane == 0) e[nb] = 1.0;
    } else {
        for (int k = lane; k < nb; k += 32) sm[k] = olde[k];
    }
    if (map32) {
        // the FP32 kernels' table of the refined map
        __syncwarp();
        const double end = refined ? 1.0 : olde[nb];
        float2* m = map32 + static_cast<int64_t>(t) * map32_stride(g) + (3 * leg + warp) * nb;
        for (int k = lane; k < nb; k += 32) m[k] = map32_value(sm[k], k + 1 < nb ? sm[k + 1] : end, warp, g);
    }
}

// The FP32 kernels' map tables of tasks [0, n_tasks) from their FP64 edges
// (edges [task][map_stride], tables [task][map32_stride]); one thread per
// entry.
__global__ void map32_kernel(Geometry g, const TaskDesc* __restrict__ tasks, int n_tasks,
                             const double* __restrict__ edges, float2* map32) {
    const int stride = map32_stride(g);
    const int64_t total = static_cast<int64_t>(n_tasks) * stride;
    for (int64_t q = blockIdx.x * static_cast<int64_t>(blockDim.x) + threadIdx.x; q < total;
         q += static_cast<int64_t>(gridDim.x) * blockDim.x) {
        const int t = static_cast<int>(q / stride), k = static_cast<int>(q - static_cast<int64_t>(t) * stride);
        const int nb = tasks[t].nbins, D = tasks[t].dim;
        if (k < D * nb)
            map32[q] = map32_entry(edges + static_cast<int64_t>(t) * g.map_stride, k / nb, k % nb, nb, g);
    }
}

// ---------------------------------------------------------------------------
// Combination of the iterations per task (inverse-variance weights; zero-
// variance iterations are exact) and assembly of Eq. (7):
// C_a(p_i) = sum_sides mult (I_gain - I_loss), err^2 = sum mult^2
// (sigma_gain^2 + sigma_loss^2).  Two lanes per (species, grid point), one for
// its gain and one for its loss tasks, 32 threads per CTA (the combination is
// a chain of FP64 divisions: spread over the SMs, 4.5 -> 3.0 us for 32 points);
// thread 0 advances the evaluation counter.
// ---------------------------------------------------------------------------
__device__ inline void combine_task(TaskAcc& A) {
    if (A.n_exact > 0.0) {
        A.mean = A.sum_exact / A.n_exact;
        A.err = 0.0;
    } else if (A.sum_inv_var > 0.0) {
        A.mean = A.sum_mean_inv_var / A.sum_inv_var;
        A.err = sqrt(1.0 / A.sum_inv_var);
    } else {
        A.mean = 0.0;
        A.err = 0.0;
    }
}

__global__ void assemble_kernel(Geometry g, const SideDesc* __restrict__ sides, TaskAcc* acc,
                                TimeState* ts, double* C, double* err, double* prev) {
    const int id = blockIdx.x * blockDim.x + threadIdx.x;
    const int k = id >> 1, term = id & 1;
    const int n = g.n_grid;
    const bool in = k < g.n_species * n;
    double c = 0.0, v = 0.0;
    const int s = in ? k / n : 0;
    const int i = in ? k - s * n : 0;
    const int nl = g.pt_hi - g.pt_lo;         // points of this context (a shard) in task order
    const bool mine = in && i >= g.pt_lo && i < g.pt_hi;
    for (int si = 0; si < g.n_side; ++si) {
        const bool here = mine && sides[si].species_obs == s;
        double mean = 0.0, e2 = 0.0;
        if (here) {
            const int t = (si * nl + i - g.pt_lo) * 2 + term;
            TaskAcc& A = acc[t];
            combine_task(A);
            if (A.mean != 0.0) prev[t] = fabs(A.mean);
            mean = A.mean;
            e2 = A.err * A.err;
        }
        const double mean1 = __shfl_xor_sync(0xffffffffu, mean, 1), e1 = __shfl_xor_sync(0xffffffffu, e2, 1);
        if (here) {
            const double mult = sides[si].mult;
            c += mult * (mean - mean1);       // (the gain lane's)
            v += mult * mult * (e2 + e1);
        }
    }
    if (in && term == 0) {
        if (!isfinite(c) || !isfinite(v)) ts->error = BEST_ERR_NUMERIC;
        C[k] = c;
        if (err) err[k] = sqrt(v);
    }
    if (id == 0) ts->call += 1u;
}

// ---------------------------------------------------------------------------
// Number and energy densities, one CTA (256 threads) per species:
//   n = Int q^2 f dq / (2 pi^2 a^3),  rho = Int q^2 E(q/a) f dq / (2 pi^2 a^3)
// over [q_min, q_max] on the FP64 not-a-knot spline (unclamped), 4-point
// Gauss-Legendre per grid interval, fixed-order tree reduction.
// ---------------------------------------------------------------------------
__global__ void moments_kernel(Geometry g, const double* __restrict__ knots, const double* __restrict__ coef64,
                               const TimeState* ts, double* n_out, double* rho_out) {
    __shared__ double sn[256], sr[256];
    const int s = blockIdx.x;
    const double a = ts->a, m = ts->mass[s];
    const double xg[4] = {-0.8611363115940526, -0.3399810435848563, 0.3399810435848563, 0.8611363115940526};
    const double wg[4] = {0.3478548451374538, 0.6521451548625461, 0.6521451548625461, 0.3478548451374538};
    double an = 0.0, ar = 0.0;
    for (int j = threadIdx.x; j < g.n_grid - 1; j += blockDim.x) {
        const double* c = coef64 + (static_cast<int64_t>(s) * (g.n_grid - 1) + j) * 4;
        const double lo = knots[j], hi = knots[j + 1];
        const double half = 0.5 * (hi - lo), mid = 0.5 * (hi + lo);
        for (int k = 0; k < 4; ++k) {
            const double q = fma(half, xg[k], mid);
            const double tt = q - lo;
            const double f = fma(fma(fma(c[3], tt, c[2]), tt, c[1]), tt, c[0]);
            const double p = q / a;
            const double wq = half * wg[k] * q * q * f;
            an += wq;
            ar += wq * sqrt(fma(p, p, m * m));
        }
    }
    sn[threadIdx.x] = an;
    sr[threadIdx.x] = ar;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            sn[threadIdx.x] += sn[threadIdx.x + h];
            sr[threadIdx.x] += sr[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double pref = 1.0 / (2.0 * kPi * kPi * a * a * a);
        n_out[s] = pref * sn[0];
        rho_out[s] = pref * sr[0];
    }
}

// ---------------------------------------------------------------------------
// Adaptive fractional width (App. C), one CTA per process after a sweep:
// r = sqrt(sum err_t^2) / sum |I_t| over the process's tasks (FP64, fixed
// summation order), then w /= factor below rel_lo, w *= factor above rel_hi,
// clamped to [w_min, w_max]; processes with a fixed width are left alone.
// ---------------------------------------------------------------------------
__global__ void width_control_kernel(Geometry g, const SideDesc* __restrict__ sides,
                                     const TaskDesc* __restrict__ tasks, const TaskAcc* __restrict__ acc,
                                     const WidthCtl* __restrict__ ctl, double* width, double* width_rel) {
    __shared__ double r2[256], ra[256];
    const int p = blockIdx.x;
    const WidthCtl c = ctl[p];
    if (c.mode != 2) return;
    double e2 = 0.0, am = 0.0;
    for (int t = threadIdx.x; t < g.n_tasks; t += blockDim.x) {
        if (sides[tasks[t].si].process != p) continue;
        const TaskAcc& A = acc[t];
        e2 = fma(A.err, A.err, e2);
        am += fabs(A.mean);
    }
    r2[threadIdx.x] = e2;
    ra[threadIdx.x] = am;
    __syncthreads();
    for (int h = blockDim.x / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            r2[threadIdx.x] += r2[threadIdx.x + h];
            ra[threadIdx.x] += ra[threadIdx.x + h];
        }
        __syncthreads();
    }
    if (threadIdx.x != 0 || !(ra[0] > 0.0)) return;
    const double rel = sqrt(r2[0]) / ra[0];
    double w = width[p];
    if (rel < c.rel_lo) w /= c.factor;
    else if (rel > c.rel_hi) w *= c.factor;
    width[p] = fmin(fmax(w, c.w_min), c.w_max);
    width_rel[p] = rel;
}

// ---------------------------------------------------------------------------
// Time stepping (Sec. 3C), one CTA of 1024 threads over all species and grid
// points.  max |C/f| is reduced in FP64 and the step used is
// dt = min(dt_requested, eps / max |C/f|) (Eq. (16)).
// ---------------------------------------------------------------------------
// Maximum of v >= 0 (not NaN) over the CTA: non-negative doubles order like
// their bits, so the reduction runs on integers (two redux operations per
// warp; an FP64 comparison takes the FP64 pipe for 64 cycles).
__device__ double warp_max_bits(double v) {
    const uint32_t hi = static_cast<uint32_t>(__double2hiint(v)), lo = static_cast<uint32_t>(__double2loint(v));
    const uint32_t mh = __reduce_max_sync(0xffffffffu, hi);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
    return __hiloint2double(static_cast<int>(mh), static_cast<int>(ml));
}
__device__ double block_max(double v, double* red) {
    v = warp_max_bits(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    v = warp_max_bits(l < static_cast<int>(blockDim.x >> 5) ? red[l] : 0.0);
    __syncthreads();
    return v;
}

// Euler (Eq. (14)) or the Heun predictor: dt from k1, logf_out = logf + dt k1/f.
// heun != 0: writes f* = exp(logf + dt k1/f) to fstar and leaves logf alone.
// The requested step is *dt_src (dt_dev itself, or the value a replayed graph
// was given).
__global__ void step_first_kernel(Geometry g, double* logf, const double* __restrict__ fgrid,
                                  const double* __restrict__ k1, double* t_dev, double* dt_dev, const double* dt_src,
                                  TimeState* ts, double* fstar, int heun) {
    __shared__ double red[32];
    const int total = g.n_species * g.n_grid;
    double mx = 0.0;
    double rate = 0.0;                       // C/f of this thread's first point
    for (int k = threadIdx.x; k < total; k += blockDim.x) {
        const double q = k1[k] / fgrid[k];
        if (k == static_cast<int>(threadIdx.x)) rate = q;
        mx = fmax(mx, fabs(q));
    }
    mx = block_max(mx, red);
    double dt = *dt_src;
    if (mx > 0.0) dt = fmin(dt, g.eps_dt / mx);
    for (int k = threadIdx.x; k < total; k += blockDim.x) {
        const double step = dt * (k == static_cast<int>(threadIdx.x) ? rate : k1[k] / fgrid[k]);
        if (heun) fstar[k] = exp(logf[k] + step);
        else logf[k] += step;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        ts->dt = dt;
        ts->t_step = *t_dev;
        if (!heun) {
            *t_dev += dt;
            *dt_dev = dt;
        }
        if (!isfinite(dt)) ts->error = BEST_ERR_NUMERIC;
    }
}

// One stage of a step from collision integrals the caller assembled (sharded
// runs), one CTA of 1024 threads; the same arithmetic as step_first_kernel
// and heun_correct_kernel with f = exp(log f).
//   stage 0: dt = min(*dt_dev, eps / max |k1/f|); Euler: log f += dt k1/f,
//            t += dt; Heun: fstar = exp(log f + dt k1/f); *dt_dev = dt.
//   stage 1 (Heun): log f += dt/2 (k1/f + k2/fstar), t += dt.
__global__ void stage_kernel(Geometry g, int heun, int stage, double* logf, const double* __restrict__ k1,
                             const double* __restrict__ k2, double* fstar, double* t_dev, double* dt_dev,
                             TimeState* ts) {
    __shared__ double red[32];
    const int total = g.n_species * g.n_grid;
    if (stage == 0) {
        double mx = 0.0;
        for (int k = threadIdx.x; k < total; k += blockDim.x) mx = fmax(mx, fabs(k1[k] / exp(logf[k])));
        mx = block_max(mx, red);
        double dt = *dt_dev;
        if (mx > 0.0) dt = fmin(dt, g.eps_dt / mx);
        for (int k = threadIdx.x; k < total; k += blockDim.x) {
            const double step = dt * k1[k] / exp(logf[k]);
            if (heun) fstar[k] = exp(logf[k] + step);
            else logf[k] += step;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            ts->dt = dt;
            ts->t_step = *t_dev;
            if (!heun) *t_dev += dt;
            *dt_dev = dt;
            if (!isfinite(dt)) ts->error = BEST_ERR_NUMERIC;
        }
    } else {
        const double dt = *dt_dev;
        for (int k = threadIdx.x; k < total; k += blockDim.x)
            logf[k] += 0.5 * dt * (k1[k] / exp(logf[k]) + k2[k] / fstar[k]);
        __syncthreads();
        if (threadIdx.x == 0) *t_dev += dt;
    }
}

// Heun corrector (Eq. (15)): logf += dt/2 (k1/f + k2/f*), f = exp(logf)
// (log f is left untouched by the predictor).
__global__ void heun_correct_kernel(Geometry g, double* logf, const double* __restrict__ fstar, const double* __restrict__ k1,
                                    const double* __restrict__ k2, double* t_dev, double* dt_dev,
                                    TimeState* ts) {
    const int total = g.n_species * g.n_grid;
    const double dt = ts->dt;
    for (int k = threadIdx.x; k < total; k += blockDim.x)
        logf[k] += 0.5 * dt * (k1[k] / exp(logf[k]) + k2[k] / fstar[k]);
    __syncthreads();
    if (threadIdx.x == 0) {
        *t_dev = ts->t_step + dt;
        *dt_dev = dt;
    }
}

}  // namespace best

// Adjoint of the fixed-sample collision integral: instantiations of the
// adjoint sample kernel and the FP64 kernels that turn its per-segment
// records and coefficient gradients into dL/df, dL/dm and dL/dcoupling.
#include <cmath>

#include "vjp_impl.cuh"

namespace best {

template <bool JVP>
void* kernel_ptr(bool f32, int nmax) {
    if (f32) {
        if (nmax <= 4) return reinterpret_cast<void*>(&vjp_kernel<float, 4, JVP>);
        if (nmax == 5) return reinterpret_cast<void*>(&vjp_kernel<float, 5, JVP>);
        return reinterpret_cast<void*>(&vjp_kernel<float, 6, JVP>);
    }
    if (nmax <= 4) return reinterpret_cast<void*>(&vjp_kernel<double, 4, JVP>);
    if (nmax == 5) return reinterpret_cast<void*>(&vjp_kernel<double, 5, JVP>);
    return reinterpret_cast<void*>(&vjp_kernel<double, 6, JVP>);
}

void* vjp_me_kernel_ptr(bool f32, int nmax, bool jvp);     // vjp_me.cu

// me: some process has an s-dependent |M|^2 (the extended instantiations)
void* vjp_kernel_ptr(bool f32, int nmax, bool me) {
    return me ? vjp_me_kernel_ptr(f32, nmax, false) : kernel_ptr<false>(f32, nmax);
}
void* jvp_kernel_ptr(bool f32, int nmax, bool me) {
    return me ? vjp_me_kernel_ptr(f32, nmax, true) : kernel_ptr<true>(f32, nmax);
}

// Adjoint seed of every task: L = sum_{a,i} v_{a,i} C~_a(p_i) and C~ = sum
// mult (I_gain - I_loss), I = K scale (sum w_n) / N, so dL/dw_n = v mult sign
// K scale / N for each of the task's samples.
__global__ void vjp_seed_kernel(Geometry g, const SideDesc* __restrict__ sides, const TaskDesc* __restrict__ tasks,
                                const TaskConst* __restrict__ tconst, const double* __restrict__ v, double* u) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.n_tasks) return;
    const TaskDesc td = tasks[t];
    const SideDesc& sd = sides[td.si];
    const double sign = td.term == 0 ? 1.0 : -1.0;
    u[t] = v[static_cast<int64_t>(sd.species_obs) * g.n_grid + td.point] * sd.mult * sign * tconst[t].K *
           tconst[t].scale / static_cast<double>(td.neval);
}

// Tangent seed: d w_n / d f_obs u_obs = (w_n / c0) dobs u_{a,i} / scale.
__global__ void jvp_seed_kernel(Geometry g, const SideDesc* __restrict__ sides, const TaskDesc* __restrict__ tasks,
                                const TaskConst* __restrict__ tconst, const SpeciesConst* __restrict__ sconst,
                                const double* __restrict__ uvec, double* u) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= g.n_tasks) return;
    const TaskDesc td = tasks[t];
    const SideDesc& sd = sides[td.si];
    const double dobs = td.term == 1 ? 1.0 : sconst[sd.species_obs].eta;
    u[t] = dobs * uvec[static_cast<int64_t>(sd.species_obs) * g.n_grid + td.point] / tconst[t].scale;
}

// Tasks of species s at grid point i in task order: f(task) for the gain and
// loss task of every side integral observed there (none outside a shard's
// points).
template <typename F>
__device__ inline void for_tasks_at(const Geometry& g, const SideDesc* __restrict__ sides, int s, int i, F&& f) {
    if (i < g.pt_lo || i >= g.pt_hi) return;
    const int nl = g.pt_hi - g.pt_lo;
    for (int si = 0; si < g.n_side; ++si) {
        if (sides[si].species_obs != s) continue;
        const int t = (si * nl + i - g.pt_lo) * 2;
        f(t);
        f(t + 1);
    }
}

// C~ and dC~ = J u from the tasks' tangent records: one thread per species
// and grid point, its tasks in task order (the same sums as one pass over all
// tasks).  A handful of dependent loads and FP64 operations per thread; one
// thread walking all tasks took 220 us for 256 tasks.
__global__ void jvp_finish_kernel(Geometry g, const SideDesc* __restrict__ sides, const TaskDesc* __restrict__ tasks,
                                  const TaskConst* __restrict__ tconst, const double* __restrict__ tot, double* C,
                                  double* JU) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= g.n_species * g.n_grid) return;
    double c = 0.0, ju = 0.0;
    for_tasks_at(g, sides, k / g.n_grid, k % g.n_grid, [&](int t) {
        const TaskDesc& td = tasks[t];
        const double* T = tot + static_cast<int64_t>(t) * 16;
        const double f = sides[td.si].mult * (td.term == 0 ? 1.0 : -1.0) * tconst[t].K * tconst[t].scale /
                         static_cast<double>(td.neval);
        c += f * T[0];
        ju += f * T[1];
    });
    C[k] = c;
    JU[k] = ju;
}

// Sum of each task's segment records in segment order, 16 doubles per task:
// 16 lanes per task, lane v summing value v, so that a record is one
// coalesced load and the chain per lane is its segments alone, eight loads in
// flight (116 us for 512 tasks when one thread summed all values of a task).
__global__ void vjp_task_kernel(Geometry g, const int32_t* __restrict__ active, const int32_t* __restrict__ task_seg,
                                const Segment* __restrict__ segs, const double* __restrict__ partials, int n_active,
                                double* tot) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    const int a = k >> 4, v = k & 15;
    if (a >= n_active) return;
    double sum = 0.0;
    if (v < 12) {
        const int s1 = task_seg[a + 1];
        int s = task_seg[a];
        for (; s + 8 <= s1; s += 8) {
            double x[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) x[u] = partials[segs[s + u].part + v];
#pragma unroll
            for (int u = 0; u < 8; ++u) sum += x[u];
        }
        for (; s < s1; ++s) sum += partials[segs[s].part + v];
    }
    tot[static_cast<int64_t>(active[a]) * 16 + v] = sum;
}

// Sum of v over the CTA (256 threads), in a fixed order.
__device__ inline double cta_sum256(double v, double* red) {
    __syncthreads();
    red[threadIdx.x] = v;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (static_cast<int>(threadIdx.x) < h) red[threadIdx.x] += red[threadIdx.x + h];
        __syncthreads();
    }
    return red[0];
}

// C~, the observed-leg and mass / coupling parts of the gradient, and the
// tail-parameter gradients per species.  CTAs [0, n_species) reduce one
// species' mass and tail gradients over all tasks, the next n_processes one
// process's coupling gradient (fixed-order tree sums), the rest take one
// (species, grid point) per thread, its tasks in task order.  (One thread
// walking all tasks took 3.0 ms for 512 tasks.)  256 threads per CTA.
__global__ void vjp_finish_kernel(Geometry g, const SideDesc* __restrict__ sides, const TaskDesc* __restrict__ tasks,
                                  const TaskConst* __restrict__ tconst, const SpeciesConst* __restrict__ sconst,
                                  const TimeState* ts, const double* __restrict__ v, const double* __restrict__ u,
                                  const double* __restrict__ tot, const double* __restrict__ coupling, double* C,
                                  double* gf, double* gm, double* gcoupling, double* gtail, int n_processes) {
    __shared__ double red[256];
    const int n = g.n_grid, S = g.n_species;
    const int b = blockIdx.x;
    auto integral = [&](int t, const TaskDesc& td) {
        const TaskConst& c = tconst[t];
        return tot[static_cast<int64_t>(t) * 16] / static_cast<double>(td.neval) * c.K * c.scale;
    };
    if (b < S) {
        double m = 0.0, tail[4] = {0.0, 0.0, 0.0, 0.0};
        for (int t = threadIdx.x; t < g.n_tasks; t += blockDim.x) {
            const SideDesc& sd = sides[tasks[t].si];
            const double* T = tot + static_cast<int64_t>(t) * 16;
            const double U = u[t];
            if (sd.species_obs == b) m += U * T[2] * ts->mass[b] / tconst[t].E_obs;
            if (sd.leg_species[sd.cons] == b) {
                m += U * T[3];
                for (int q = 0; q < 4; ++q) tail[q] += U * T[4 + q];
            }
            for (int j = 0; j < sd.n - 2; ++j)
                if (sd.leg_species[sd.integ[j]] == b) m += U * T[8 + j];
        }
        m = cta_sum256(m, red);
        if (threadIdx.x == 0) gm[b] = m;
        for (int q = 0; q < 4; ++q) {
            const double x = cta_sum256(tail[q], red);
            if (threadIdx.x == 0) gtail[b * 4 + q] = x;
        }
        return;
    }
    if (b < S + n_processes) {
        const int p = b - S;
        double l = 0.0;
        for (int t = threadIdx.x; t < g.n_tasks; t += blockDim.x) {
            const TaskDesc& td = tasks[t];
            const SideDesc& sd = sides[td.si];
            if (sd.process != p) continue;
            const double sign = td.term == 0 ? 1.0 : -1.0;
            l += 2.0 / coupling[p] * sd.mult * sign * integral(t, td) *
                 v[static_cast<int64_t>(sd.species_obs) * n + td.point];
        }
        l = cta_sum256(l, red);
        if (threadIdx.x == 0) gcoupling[p] = l;
        return;
    }
    const int k = (b - S - n_processes) * blockDim.x + threadIdx.x;
    if (k >= S * n) return;
    const int a = k / n;
    double c = 0.0, gr = 0.0;
    for_tasks_at(g, sides, a, k - a * n, [&](int t) {
        const TaskDesc& td = tasks[t];
        const double dobs = td.term == 1 ? 1.0 : sconst[a].eta;
        c += sides[td.si].mult * (td.term == 0 ? 1.0 : -1.0) * integral(t, td);
        gr += u[t] * tot[static_cast<int64_t>(t) * 16 + 1] * dobs / tconst[t].scale;
    });
    C[k] = c;
    gf[k] = gr;
}

}  // namespace best

// pd_step_verlet: FCBM-EC dynamics with energy-based bond breaking.
//
// Per step (Eq. 83-84 for the kinematics, Eq. 63 for the integrity index,
// Eq. 101-102 for L and W with node weight chi_B lam):
//   kick+drift : v <- v + dt/(2 rho) (L^n + b);  u <- chi_O (u + dt v) + (1 - chi_O) w;
//                lam <- lam [W^n <= Wc]  (irreversible; counts 1 -> 0 flips)
//   G^lam      : recomputed on the device only if some lam flipped this step
//   force      : L^{n+1}, W^{n+1} = FFT convolutions with weight chi_B lam
//   kick       : v <- chi_O (v + dt/(2 rho) (L^{n+1} + b))
// The call starts with one force evaluation of the given state, so a run of
// n steps split over several calls gives the same result as one call.
//
// Energy mode 1 (pd_plan_set_energy_mode) evaluates W of Eq. 102 by the plain
// horizon sum of Eq. 47 instead of the three convolutions T1 - 2 u.(C*(v u))
// + u.(C*v) u: the convolutions' rounding error is global, about
// eps lambda_max (rms|u|^2 + 2 |u(x)| rms|u|) at every node, which in FP32
// exceeds Wc once fragments have moved far (|u| ~ 10-100 grid units), while
// the direct sum errs by about eps |u(x)| / |eta| relative to W, locally.
#include <algorithm>
#include <cmath>

#include "pd_horizon.cuh"
#include "pd_ops.cuh"
#include "pd_plan.cuh"

namespace pd {

template <typename T>
pd_status force_any(pd_plan *p, const T *u, const T *s, const uint8_t *lam, const T *G, T *L, T *W,
                    cudaStream_t st);

namespace {

// device counters live in the reduction buffer; the change flag of step s is
// changed[s & 1], cleared by the step before
struct VerletCounters {
    unsigned long long flips;
    int changed[2];
};

// First kick, drift and integrity update of step s; with `kick` the second kick
// of the step before comes first (the force L is the same for both), so that a
// run of steps reads L, b and v once per step.
// Gamma values at the end of the step: w + t_next w1 (w1 null: w, constant)
// One node per thread and all loads ahead of the first store: with a few nodes
// in series per thread and the components one after the other the kernel waited
// for memory most of its 10.8 us (1024 x 512; now 6.7).
template <typename T, int D>
__global__ void __launch_bounds__(256) k_kick_drift(T *u, T *v, uint8_t *lam, const T *L, const T *b, const T *w,
                                                    const T *w1, T t_next, const T *W, const uint8_t *chi,
                                                    const uint8_t *co, int64_t N, T hdt_rho, T dt, T Wc,
                                                    int breaking, int kick, int s, VerletCounters *cnt)
{
    unsigned long long flips = 0;
    if (blockIdx.x == 0 && threadIdx.x == 0) cnt->changed[(s + 1) & 1] = 0;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p < N) {
        T a[D], vn[D], un[D], g[D];
        bool on[D];
        bool whole = false;
        T Wp = T(0);
        if (breaking) {
            whole = (chi[p] != 0) & (lam[p] != 0);
            Wp = W[p];
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const int64_t q = i * N + p;
            a[i] = hdt_rho * (L[q] + b[q]);
            on[i] = co[q] != 0;
            vn[i] = v[q];
            un[i] = u[q];
            g[i] = w ? w[q] : T(0);
            if (w1) g[i] = g[i] + t_next * w1[q];
        }
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const int64_t q = i * N + p;
            if (kick) vn[i] = on[i] ? vn[i] + a[i] : T(0);
            const T vh = vn[i] + a[i];
            v[q] = vh;
            u[q] = on[i] ? un[i] + dt * vh : g[i];
        }
        if (whole && !(Wp <= Wc)) {
            lam[p] = 0;
            ++flips;
        }
    }
    // warp-aggregated counter update
    for (int o = 16; o > 0; o >>= 1) flips += __shfl_down_sync(0xffffffffu, flips, o);
    if ((threadIdx.x & 31) == 0 && flips) {
        atomicAdd(&cnt->flips, flips);
        atomicExch(&cnt->changed[s & 1], 1);
    }
}

template <typename T>
__global__ void k_kick(T *v, const T *L, const T *b, const uint8_t *co, int64_t n, T hdt_rho)
{
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x)
        v[q] = co[q] ? v[q] + hdt_rho * (L[q] + b[q]) : T(0);
}

// W(x) = 1/2 chi lam Σ_H chi' lam' eta.C(xi).eta dV, eta = u(x+xi) - u(x)
// (Eq. 47 with the integrity weights of Eq. 44; periodic neighbour offsets).
// The bond tensor is rank one, C(xi) dV = c(xi) xi xi^T / |xi|^2 with
// c = tr C dV, so each bond adds c (xi.eta)^2 / |xi|^2: the projection is
// formed first, and a rigidly rotating neighbourhood (large eta nearly
// normal to xi) does not cancel large quadratic-form terms.
template <typename T, int D>
__global__ void k_energy_direct(int n1, int n2, int n3, HorizonDev hz, double dx1, double dx2, double dx3,
                                const uint8_t *chi, const uint8_t *lam, const T *u, T *W, int64_t N)
{
    constexpr int NC = Sym<D>::n;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T *ws = reinterpret_cast<T *>(sm_raw);            // cnt: c / |xi|^2
    T *xs = ws + hz.cnt;                               // D x cnt: xi
    int *os = reinterpret_cast<int *>(xs + D * hz.cnt);  // 3 x cnt
    for (int c = threadIdx.x; c < hz.cnt; c += blockDim.x) {
        const double x[3] = {hz.off[3 * c] * dx1, hz.off[3 * c + 1] * dx2, hz.off[3 * c + 2] * dx3};
        double tr = 0.0, r2 = 0.0;
        for (int k = 0; k < NC; ++k)
            if (Sym<D>::i(k) == Sym<D>::j(k)) tr += hz.c[k * hz.cnt + c];
        for (int j = 0; j < D; ++j) r2 += x[j] * x[j];
        ws[c] = (T)(tr / r2);
        for (int j = 0; j < D; ++j) xs[j * hz.cnt + c] = (T)x[j];
        for (int j = 0; j < 3; ++j) os[3 * c + j] = hz.off[3 * c + j];
    }
    __syncthreads();
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < N; p += (int64_t)gridDim.x * blockDim.x) {
        T acc = T(0);
        if (chi[p] && lam[p]) {
            int i1, i2, i3;
            node_coords(p, n1, n2, i1, i2, i3);
            T up[D];
#pragma unroll
            for (int j = 0; j < D; ++j) up[j] = u[j * N + p];
            for (int c = 0; c < hz.cnt; ++c) {
                const int a = (i1 + os[3 * c]) & (n1 - 1);
                const int b = (i2 + os[3 * c + 1]) & (n2 - 1);
                const int e = (i3 + os[3 * c + 2]) & (n3 - 1);
                const int64_t q = ((int64_t)e * n2 + b) * n1 + a;
                if (!(chi[q] && lam[q])) continue;
                T s = T(0);
#pragma unroll
                for (int j = 0; j < D; ++j) s += xs[j * hz.cnt + c] * (u[j * N + q] - up[j]);
                acc += ws[c] * s * s;
            }
        }
        W[p] = T(0.5) * acc;
    }
}

// One column of bonds of the same sum (pd_horizon.cuh). MASK: neighbours whose
// weight is 0 add nothing; without it the whole tile has weight 1.
template <typename T, int D, int Z, bool MASK>
__device__ __forceinline__ void energy_column(const T *tu, const uint8_t *tm, int tile, const T *bond, int e, int step,
                                              int rc, const T (&up)[kNodes][D], T (&acc)[kNodes])
{
    T a[kNodes + 2 * Z][D];
    bool in[kNodes + 2 * Z];
#pragma unroll
    for (int z = 0; z < kNodes + 2 * Z; ++z) {
#pragma unroll
        for (int j = 0; j < D; ++j) a[z][j] = tu[j * tile + e + (z - Z) * step];
        in[z] = !MASK || tm[e + (z - Z) * step];
    }
#pragma unroll
    for (int oc = -Z; oc <= Z; ++oc) {
        T x[D];
#pragma unroll
        for (int j = 0; j < D; ++j) x[j] = bond[4 * (rc + oc) + j];
        const T w = bond[4 * (rc + oc) + 3];
#pragma unroll
        for (int m = 0; m < kNodes; ++m) {
            T s = T(0);
#pragma unroll
            for (int j = 0; j < D; ++j) s += x[j] * (a[m + Z + oc][j] - up[m][j]);
            const T next = acc[m] + w * s * s;
            acc[m] = in[m + Z + oc] ? next : acc[m];
        }
    }
}

// The same sum on shared-memory tiles, column by column; the column of the
// node itself has weight 0 at oc = 0. Tiles entirely of weight 1 (most of a
// body) take the loop without masks.
template <typename T, int D>
__global__ void __launch_bounds__(kHzX *kHzY)
    k_energy_tile(HzTile t, HzTables<T> tab, const uint8_t *__restrict__ chi, const uint8_t *__restrict__ lam,
                  const T *__restrict__ u, T *__restrict__ W, int64_t N)
{
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T *bond = reinterpret_cast<T *>(sm_raw);  // [columns][2 rc + 1][4]: xi, c / |xi|^2
    const int nz = 2 * t.rc + 1, slots = t.ncol * nz;
    int2 *col = reinterpret_cast<int2 *>(bond + 4 * slots);
    T *tu = reinterpret_cast<T *>(col + ((t.ncol + 1) & ~1));  // [D][tile], 0 where the weight is 0
    const int tile = t.p * t.rows * t.nz;
    uint8_t *tm = reinterpret_cast<uint8_t *>(tu + (size_t)D * tile);  // weight mask
    const int tid = threadIdx.y * kHzX + threadIdx.x;
    for (int c = tid; c < slots; c += kHzX * kHzY) {
#pragma unroll
        for (int k = 0; k < 4; ++k) bond[4 * c + k] = tab.bond[4 * c + k];
    }
    for (int c = tid; c < t.ncol; c += kHzX * kHzY) col[c] = tab.col[t.ncol + c];
    bool all = true;
    hz_fill(t, [&](int e, int64_t q) {
        const bool in = chi[q] != 0 && lam[q] != 0;
        T x[D];
#pragma unroll
        for (int j = 0; j < D; ++j) x[j] = u[j * N + q];
        all = all && in;
        tm[e] = in ? 1 : 0;
#pragma unroll
        for (int j = 0; j < D; ++j) tu[j * tile + e] = in ? x[j] : T(0);
    });
    const bool full = __syncthreads_and(all);
    const int e0 = hz_elem0(t);
    T up[kNodes][D], acc[kNodes];
#pragma unroll
    for (int m = 0; m < kNodes; ++m) {
        acc[m] = T(0);
#pragma unroll
        for (int j = 0; j < D; ++j) up[m][j] = tu[j * tile + e0 + m * t.step];
    }
    const int *grp = tab.grp + kHzReach + 2;
#define PD_ENERGY_COLUMNS(Z, MASK)                                                                       \
    _Pragma("unroll 1") for (int c = __ldg(grp + Z); c < __ldg(grp + Z + 1); ++c)                         \
    {                                                                                                    \
        const int2 k = col[c];                                                                           \
        energy_column<T, D, Z, MASK>(tu, tm, tile, bond + 4 * k.y, e0 + k.x, t.step, t.rc, up, acc);     \
    }
    if (full) {
        PD_ENERGY_COLUMNS(0, false)
        PD_ENERGY_COLUMNS(1, false)
        PD_ENERGY_COLUMNS(2, false)
        PD_ENERGY_COLUMNS(3, false)
        PD_ENERGY_COLUMNS(4, false)
    } else {
        PD_ENERGY_COLUMNS(0, true)
        PD_ENERGY_COLUMNS(1, true)
        PD_ENERGY_COLUMNS(2, true)
        PD_ENERGY_COLUMNS(3, true)
        PD_ENERGY_COLUMNS(4, true)
    }
#undef PD_ENERGY_COLUMNS
#pragma unroll
    for (int m = 0; m < kNodes; ++m) {
        int64_t p;
        if (hz_node(t, m, p)) W[p] = tm[e0 + m * t.step] ? T(0.5) * acc[m] : T(0);
    }
}

template <typename T>
pd_status energy_direct(pd_plan *p, const T *u, const uint8_t *lam, T *W, cudaStream_t st)
{
    const int cnt = p->hdev.cnt;
    {
        const HzTile t = hz_tile(p->dim, p->n1, p->n2, p->n3, p->hdev);
        const size_t ts = (size_t)4 * t.ncol * (2 * t.rc + 1) * sizeof(T) +
                          (size_t)((t.ncol + 1) & ~1) * sizeof(int2) +
                          (size_t)t.p * t.rows * t.nz * (p->dim * sizeof(T) + 1);
        if (ts <= kHzSmem && t.rc <= kHzReach && p->hzcol) {
            const auto kern = p->dim == 3 ? k_energy_tile<T, 3> : k_energy_tile<T, 2>;
            PD_TRY(set_smem_attr((const void *)kern, ts));
            kern<<<hz_grid(t), dim3(kHzX, kHzY), ts, st>>>(t, hz_tables<T>(p, t), p->chi, lam, u, W, p->N);
            PD_LAUNCH_CHECK();
            p->launches++;
            return PD_OK;
        }
    }
    const size_t smem = (size_t)(1 + p->dim) * cnt * sizeof(T) + (size_t)3 * cnt * sizeof(int);
    const double *dx = p->prob.dx;
    const unsigned ng = (unsigned)std::min<int64_t>(8 * p->nsm, (p->N + 255) / 256);
    if (p->dim == 3) {
        PD_TRY(set_smem_attr((const void *)k_energy_direct<T, 3>, smem));
        k_energy_direct<T, 3><<<ng, 256, smem, st>>>(p->n1, p->n2, p->n3, p->hdev, dx[0], dx[1], dx[2], p->chi, lam,
                                                     u, W, p->N);
    } else {
        PD_TRY(set_smem_attr((const void *)k_energy_direct<T, 2>, smem));
        k_energy_direct<T, 2><<<ng, 256, smem, st>>>(p->n1, p->n2, p->n3, p->hdev, dx[0], dx[1], dx[2], p->chi, lam,
                                                     u, W, p->N);
    }
    PD_LAUNCH_CHECK();
    p->launches++;
    return PD_OK;
}

// one force evaluation of the step, with W in the plan's energy mode
template <typename T>
pd_status step_force(pd_plan *p, const T *u, const uint8_t *lam, const T *G, T *L, T *W, int breaking,
                     cudaStream_t st)
{
    if (breaking && p->energy_direct) {
        PD_TRY(force_any<T>(p, u, nullptr, lam, G, L, nullptr, st));
        return energy_direct<T>(p, u, lam, W, st);
    }
    return force_any<T>(p, u, nullptr, lam, G, L, breaking ? W : nullptr, st);
}

template <typename T>
pd_status verlet_impl(pd_plan *p, T *u, T *v, uint8_t *lam, const T *b, const T *w, const T *w1, double t0,
                      double dt, int nsteps, int64_t *n_broken_out, cudaStream_t st)
{
    const int d = p->dim;
    const int64_t N = p->N;
    T *L = (T *)p->cg_q;
    T *W = (T *)p->theta;
    T *G = lam ? (T *)p->Gw : (sizeof(T) == 8 ? (T *)p->G64 : (T *)p->G32);
    const int breaking = (lam && p->wc > 0) ? 1 : 0;
    VerletCounters *cnt = reinterpret_cast<VerletCounters *>(p->red + kRedVerlet);
    PD_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(VerletCounters), st));
    if (lam) {
        PD_TRY((launch_gfield<T, uint8_t>(p, lam, G, nullptr, st)));
        p->launches++;
    }
    PD_TRY(step_force<T>(p, u, lam, G, L, W, breaking, st));
    const T hdt = (T)(0.5 * dt / p->prob.rho);
    const auto kick_drift = d == 3 ? k_kick_drift<T, 3> : k_kick_drift<T, 2>;
    const unsigned nblk = (unsigned)((N + 255) / 256);
    const unsigned ngv = (unsigned)std::min<int64_t>(4 * p->nsm, (d * N + 255) / 256);
    for (int s = 0; s < nsteps; ++s) {
        const T t_next = (T)(t0 + (double)(s + 1) * dt);
        kick_drift<<<nblk, 256, 0, st>>>(u, v, lam, L, b, w, w1, t_next, W, p->chi, p->chi_om, N, hdt, (T)dt,
                                         (T)p->wc, breaking, s > 0 ? 1 : 0, s, cnt);
        PD_LAUNCH_CHECK();
        p->launches++;
        if (breaking) {
            // G^lam, skipped unless this step's kick-drift flagged a change
            PD_TRY((launch_gfield<T, uint8_t>(p, lam, G, &cnt->changed[s & 1], st)));
            p->launches++;
        }
        PD_TRY(step_force<T>(p, u, lam, G, L, W, breaking, st));
    }
    if (nsteps > 0) {
        k_kick<T><<<ngv, 256, 0, st>>>(v, L, b, p->chi_om, d * N, hdt);
        PD_LAUNCH_CHECK();
        p->launches++;
    }
    if (n_broken_out) {
        VerletCounters h;
        PD_CUDA_TRY(cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, st));
        PD_CUDA_TRY(cudaStreamSynchronize(st));
        *n_broken_out = (int64_t)h.flips;
    }
    return PD_OK;
}

}  // namespace
}  // namespace pd

using namespace pd;

static pd_status verlet_entry(pd_plan *p, void *u, void *v, uint8_t *lambda, const void *b, const void *w,
                              const void *w1, double t0, double dt, int nsteps, int64_t *n_broken_out, void *stream,
                              const char *who)
{
    if (!p || !u || !v || !b) {
        set_error("%s: null plan, u, v or b", who);
        return PD_ERR_ARG;
    }
    if (!(dt > 0) || nsteps < 0 || !(p->prob.rho > 0) || !std::isfinite(t0)) {
        set_error("%s: dt and rho must be positive, nsteps >= 0, t0 finite", who);
        return PD_ERR_ARG;
    }
    if (p->state_based || p->nonlinear) {
        set_error("%s: the dynamic driver uses the linearized bond model", who);
        return PD_ERR_ARG;
    }
    cudaStream_t st = (cudaStream_t)stream;
    if (p->prob.fp64)
        return verlet_impl<double>(p, (double *)u, (double *)v, lambda, (const double *)b, (const double *)w,
                                   (const double *)w1, t0, dt, nsteps, n_broken_out, st);
    return verlet_impl<float>(p, (float *)u, (float *)v, lambda, (const float *)b, (const float *)w,
                              (const float *)w1, t0, dt, nsteps, n_broken_out, st);
}

extern "C" pd_status pd_step_verlet(pd_plan *p, void *u, void *v, uint8_t *lambda, const void *b, const void *w,
                                    double dt, int nsteps, int64_t *n_broken_out, void *stream)
{
    return verlet_entry(p, u, v, lambda, b, w, nullptr, 0.0, dt, nsteps, n_broken_out, stream, "pd_step_verlet");
}

extern "C" pd_status pd_step_verlet_ramp(pd_plan *p, void *u, void *v, uint8_t *lambda, const void *b,
                                         const void *w0, const void *w1, double t0, double dt, int nsteps,
                                         int64_t *n_broken_out, void *stream)
{
    if (!w1) {
        set_error("pd_step_verlet_ramp: w1 is required (use pd_step_verlet for a constant w)");
        return PD_ERR_ARG;
    }
    return verlet_entry(p, u, v, lambda, b, w0, w1, t0, dt, nsteps, n_broken_out, stream, "pd_step_verlet_ramp");
}

extern "C" pd_status pd_plan_set_energy_mode(pd_plan *p, int mode)
{
    if (!p || (mode != 0 && mode != 1)) {
        set_error("pd_plan_set_energy_mode: null plan or mode not 0/1");
        return PD_ERR_ARG;
    }
    p->energy_direct = mode;
    return PD_OK;
}

// pd_force: one FCBM-EC force evaluation as fused FFT-convolution passes.
//
// Bond model (Eq. 57-58, 75, 100-102), d = 2 or 3, node weight v = chi s:
//   rows   : X_j = FFT_x1(v u_j)            [+ Q_ij = FFT_x1(v u_i u_j) for W]
//   cols   : FFT_x2                          (3D only)
//   last   : FFT_x3 (3D) / FFT_x2 (2D), Y_i = M^_ij X_j [, T = Σ M^_ij Q_ij], inverse
//   cols   : inverse FFT_x2                  (3D only)
//   rows   : inverse FFT_x1, L_i = v (y_i - G_ij u_j) [, W]
// State-based model with 3 kappa != 5 mu (Eq. 92, 95-97) adds the dilatation
// round trip between the two halves (see force_state below).
#pragma once
#include "pd_horizon.cuh"
#include "pd_ops.cuh"

namespace pd {

// Fit of the affine split (pd_affine.cuh): block sums over the body, then the
// exact-form coefficients in the plan's coefficient buffer.
template <typename T, int D>
pd_status affine_fit(pd_plan *p, const T *u, cudaStream_t st, AffineView<T> *view)
{
    constexpr int kBlocks = 296;  // 2 x 148 SMs' worth; the sums are a small part of the evaluation
    AffFitArgs fa;
    for (int i = 0; i < 16; ++i) fa.inv[i] = p->aff_inv[i];
    for (int k = 0; k < 3; ++k) fa.emax[k] = p->aff_emax[k];
    fa.nblk = kBlocks;
    const int lg1 = ilog2(p->n1), lg2 = ilog2(p->n2);
    PD_TRY(launch_k(p->pdl != 0, k_aff_sums<T, D>, dim3(kBlocks), dim3(256), 0, st, u, (const uint8_t *)p->chi, lg1,
                    lg2, p->aff_c[0], p->aff_c[1], p->aff_c[2], p->N, p->red));
    T *coef = reinterpret_cast<T *>(p->aff_coef);
    PD_TRY(launch_k(p->pdl != 0, k_aff_fit<T, D>, dim3(1), dim3(256), 0, st, (const double *)p->red, fa, coef));
    p->launches += 2;
    *view = AffineView<T>{coef, p->aff_c[0], p->aff_c[1], p->aff_c[2], lg1, lg2};
    return PD_OK;
}

// Weight chi_B (s = lam = null) or chi_B s or chi_B lam. G null: the epilogue
// takes the plan's boundary-node list (weight chi_B only), else the dense G of
// the weight. aff: transform u - a, a the affine fit (list only, no energy).
template <typename T, int D, bool ENERGY>
pd_status force_bond_pipeline(pd_plan *p, const T *u, const T *s, const uint8_t *lam, const T *G, T *L, T *W,
                              cudaStream_t st, bool aff = false)
{
    cx<T> *spec = reinterpret_cast<cx<T> *>(spec_buf<T>(p));
    const int64_t fs = p->N / 2;
    constexpr int FI = D + (ENERGY ? Sym<D>::n : 0), FO = D + (ENERGY ? 1 : 0);
    PD_TRY(check_slots<T>(p, FI));
    AffineView<T> av{};
    if (aff) PD_TRY((affine_fit<T, D>(p, u, st, &av)));
    const NodeWeight<T> w{s, lam};
    ProForce<T, D, ENERGY> pro{u, w, p->chi, p->N, p->n1, spec, fs, av};
    PD_TRY(launch_rows<T>(p, pro, st));
    if (D == 3) PD_TRY(col_pass<T>(p, 0, FI, false, st));
    CombForce<T, D, ENERGY> cmb{model_view<T>(p)};
    PD_TRY(launch_comb<T>(p, cmb, st));
    if (D == 3) PD_TRY(col_pass<T>(p, 0, FO, true, st));
    if (!G) {
        const Model<T> m = model_view<T>(p);
        EpiForceSparse<T, D, ENERGY> epi{u, p->chi, m.gent, p->goff, L, W, p->N, p->n1, spec, fs, av,
                                         reinterpret_cast<const T *>(p->aff_tab)};
        return launch_rows<T>(p, epi, st);
    }
    EpiForceDense<T, D, ENERGY> epi{u, w, p->chi, G, L, W, p->N, p->n1, spec, fs};
    return launch_rows<T>(p, epi, st);
}

// ---------------------------------------------------------------------------
// State-based solid with dilatation (3D). With g_i = omega xi_i, the plan's
// node field q_i(x) = Σ_H g_i dV chi(x+xi) = -dV (g_i * chi)(x), and the
// correlation Σ_H g_i f(x+xi) dV = -dV (g_i * f)(x) (g is odd):
//   theta = (3 chi / m) Σ chi' omega xi.(u' - u) dV
//         = -(3 chi / m) [ dV g_i*(chi u_i) + q_i u_i ]                   (Eq. 93, 96)
//   L_i   = chi [ conv_M(chi u)_i - G_ij u_j + ka theta q_i - ka dV g_i*theta ]  (Eq. 92, 95)
// with ka = (3 kappa - 5 mu)/m0. The spectrum of g_i is -i gamma_i with
// gamma_i = Σ g_i sin(theta) (odd), so FFT(dV g_i * f)/N = -i ghat_i FFT(f),
// ghat_i = dV gamma_i / N.
// ---------------------------------------------------------------------------

// Slots: 0-2 chi u_j (x1, x2 transformed), 3 S, 4 theta; 0-2 again for the
// outputs. The second combine transforms chi u_j along x3 once more: cheaper
// than writing three transformed spectra and reading them back.
// last axis, first combine: S = Σ -i ghat_i X_i
template <typename T>
struct CombTheta {
    static constexpr int kFin = 3, kFout = 1, kTab = 3, kDim = 3;
    Model<T> m;
    __device__ int slot_in(int f) const { return f; }
    __device__ int slot_out(int) const { return 3; }
    __device__ const T *table(int c) const { return m.ghat + c * m.fold_sz; }
    __device__ __forceinline__ void combine(const T *t, bool fy, bool fz, const cx<T> *in, cx<T> *out) const
    {
        T g[3];
        load_ghat_s(t, fy, fz, g);
        cx<T> acc = mk(T(0), T(0));
#pragma unroll
        for (int i = 0; i < 3; ++i) acc = acc + scale(in[i], g[i]);
        out[0] = mk(acc.y, -acc.x);  // -i acc
    }
};

// rows: inverse of S, theta at the nodes, forward transform of theta
template <typename T>
struct RowTheta {
    static constexpr int kFin = 1, kFout = 1, kNB = 0, kDim = 3;
    Model<T> m;
    const T *u;
    T *theta;
    cx<T> *spec;
    int64_t fstride;
    __device__ const cx<T> *spec_in(int) const { return spec + 3 * fstride; }
    __device__ cx<T> *spec_out(int) const { return spec + 4 * fstride; }
    __device__ const uint8_t *nb_src(int) const { return nullptr; }
    struct Nd {
        T ma, mb, ga[3], gb[3], ua[3], ub[3];
        uchar2 in;
    };
    __device__ __forceinline__ void load(Nd &nd, int64_t p0, int o) const
    {
        load_pair(m.m3inv + p0 + o, nd.ma, nd.mb);
        nd.in = *reinterpret_cast<const uchar2 *>(m.chi + p0 + o);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            load_pair(m.qt + (i * m.N + p0) + o, nd.ga[i], nd.gb[i]);
            load_pair(u + (i * m.N + p0) + o, nd.ua[i], nd.ub[i]);
        }
    }
    __device__ __forceinline__ void node2(const RowCtx &c, int o, Nd &nd, const T *in0, const T *in1, T *o0,
                                          T *o1, DSum &) const
    {
        T qa = T(0), qb = T(0);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            qa += nd.ga[i] * nd.ua[i];
            qb += nd.gb[i] * nd.ub[i];
        }
        const T t0 = nd.in.x ? -nd.ma * (in0[0] + qa) : T(0), t1 = nd.in.y ? -nd.mb * (in1[0] + qb) : T(0);
        store2(theta + c.p0 + o, t0, t1);
        o0[0] = t0;
        o1[0] = t1;
    }
    __device__ void block_done(DSum &) const {}
};

// last axis, second combine: Y_i = M^_ij X_j + i ka ghat_i Theta
template <typename T>
struct CombState {
    static constexpr int kFin = 4, kFout = 3, kTab = 9, kDim = 3;
    Model<T> m;
    __device__ int slot_in(int f) const { return f < 3 ? f : 4; }
    __device__ int slot_out(int f) const { return f; }
    __device__ const T *table(int c) const { return c < 6 ? m.mhat + c * m.fold_sz : m.ghat + (c - 6) * m.fold_sz; }
    __device__ __forceinline__ void combine(const T *t, bool fy, bool fz, const cx<T> *in, cx<T> *out) const
    {
        T M[9], g[3];
        load_mhat_s(3, t, fy, fz, M);
        load_ghat_s(t + 6, fy, fz, g);
        mat_vec<T, 3>(M, in, out);
        const cx<T> it = mul_i(in[3]);
#pragma unroll
        for (int i = 0; i < 3; ++i) out[i] = out[i] + scale(it, m.ka * g[i]);
    }
};

// rows: inverse of Y, L = chi y, boundary nodes:
//   L_i -= G_ij u_j - ka theta q_i   (q_i and G vanish off the boundary list)
template <typename T>
struct EpiState {
    static constexpr int kFin = 3, kFout = 0, kNB = 1, kDim = 3;
    static constexpr bool kEntries = true;
    Model<T> m;
    const T *u;
    const T *theta;
    T *L;
    const cx<T> *spec;
    int64_t fstride;
    __device__ const cx<T> *spec_in(int f) const { return spec + f * fstride; }
    __device__ cx<T> *spec_out(int) const { return nullptr; }
    __device__ const uint8_t *nb_src(int) const { return m.chi; }
    __device__ __forceinline__ const int *rows_off() const { return m.goff; }
    __device__ __forceinline__ void entry(int k, int64_t &p, T *s) const
    {
        const GEntry<T> e = m.gent[k];
        p = e.p;
        T uu[3], Gu[3] = {T(0), T(0), T(0)};
#pragma unroll
        for (int j = 0; j < 3; ++j) uu[j] = u[j * m.N + p];
        sym_apply<T, 3>(e.g, uu, Gu);
        const T th = theta[p];
#pragma unroll
        for (int i = 0; i < 3; ++i) s[i] = m.ka * th * m.qt[i * m.N + p] - Gu[i];
    }
    struct Nd {
    };
    __device__ __forceinline__ void load(Nd &, int64_t, int) const {}
    __device__ __forceinline__ void node2(const RowCtx &c, int o, Nd &, const T *in0, const T *in1, T *, T *,
                                          DSum &) const
    {
        const uchar2 b = c.b2(0, o);
#pragma unroll
        for (int i = 0; i < 3; ++i) store2(L + (i * m.N + c.p0) + o, b.x ? in0[i] : T(0), b.y ? in1[i] : T(0));
    }
    __device__ void block_done(DSum &) const {}
};

template <typename T>
pd_status force_state_pipeline(pd_plan *p, const T *u, T *L, T *theta, cudaStream_t st)
{
    cx<T> *spec = reinterpret_cast<cx<T> *>(spec_buf<T>(p));
    const int64_t fs = p->N / 2;
    const Model<T> m = model_view<T>(p);
    PD_TRY(check_slots<T>(p, 5));
    ProForce<T, 3, false> pro{u, NodeWeight<T>{nullptr, nullptr}, p->chi, p->N, p->n1, spec, fs, AffineView<T>{}};
    PD_TRY(launch_rows<T>(p, pro, st));
    PD_TRY(col_pass<T>(p, 0, 3, false, st));
    CombTheta<T> c1{m};
    PD_TRY(launch_comb<T>(p, c1, st));
    PD_TRY(col_pass<T>(p, 3, 1, true, st));
    RowTheta<T> rt{m, u, theta, spec, fs};
    PD_TRY(launch_rows<T>(p, rt, st));
    PD_TRY(col_pass<T>(p, 4, 1, false, st));
    CombState<T> c2{m};
    PD_TRY(launch_comb<T>(p, c2, st));
    PD_TRY(col_pass<T>(p, 0, 3, true, st));
    EpiState<T> epi{m, u, theta, L, spec, fs};
    PD_TRY(launch_rows<T>(p, epi, st));
    return PD_OK;
}

// Boundary field for a node weight (s and/or lam): G = conv_M(chi s lam), direct sum.
template <typename T>
pd_status weight_gfield(pd_plan *p, const T *s, const uint8_t *lam, T *G, cudaStream_t st)
{
    if (s && lam) {
        set_error("weight_gfield: s and lambda together are not supported");
        return PD_ERR_ARG;
    }
    if (s)
        PD_TRY((launch_gfield<T, T>(p, s, G, nullptr, st)));
    else
        PD_TRY((launch_gfield<T, uint8_t>(p, lam, G, nullptr, st)));
    p->launches++;
    return PD_OK;
}

// Bond-model force with weight chi_B (s = lam = null: sparse plan G), chi_B s
// or chi_B lam (dense G of that weight passed in G).
template <typename T>
pd_status force_any(pd_plan *p, const T *u, const T *s, const uint8_t *lam, const T *G, T *L, T *W,
                    cudaStream_t st)
{
    if (s && lam) {
        set_error("force: s and lambda together are not supported");
        return PD_ERR_ARG;
    }
    const T *g = s || lam ? G : nullptr;  // weight chi_B: the plan's list
    if (p->dim == 2) {
        if (W) return force_bond_pipeline<T, 2, true>(p, u, s, lam, g, L, W, st);
        return force_bond_pipeline<T, 2, false>(p, u, s, lam, g, L, W, st);
    }
    if (W) return force_bond_pipeline<T, 3, true>(p, u, s, lam, g, L, W, st);
    return force_bond_pipeline<T, 3, false>(p, u, s, lam, g, L, W, st);
}

template <typename T>
T *work_theta(pd_plan *p)
{
    if constexpr (sizeof(T) == 8) {
        if (!p->prob.fp64) return reinterpret_cast<T *>(p->theta64);
    }
    return reinterpret_cast<T *>(p->theta);
}

template <typename T>
pd_status force_plain(pd_plan *p, const T *u, const T *s, T *L, T *W, cudaStream_t st)
{
    if (p->state_based) {
        if (s || W) {
            set_error("pd_force: node weight and energy output are for the bond model only");
            return PD_ERR_ARG;
        }
        return force_state_pipeline<T>(p, u, L, work_theta<T>(p), st);
    }
    const T *G = sizeof(T) == 8 ? (const T *)p->G64 : (const T *)p->G32;
    if (s) {
        if (sizeof(T) == 8 && !p->prob.fp64) {
            set_error("pd_force: FP64 node weight on an FP32 plan is not supported");
            return PD_ERR_ARG;
        }
        T *Gs = reinterpret_cast<T *>(p->Gw);
        PD_TRY(weight_gfield<T>(p, s, nullptr, Gs, st));
        G = Gs;
    }
    return force_any<T>(p, u, s, nullptr, G, L, W, st);
}

// pd_force: force_plain, or with the affine split when the plan has it on and
// the call is the plain bond force in the plan's precision (pd_affine.cuh)
template <typename T>
pd_status force_public(pd_plan *p, const T *u, const T *s, T *L, T *W, cudaStream_t st)
{
    const bool aff = p->affine_split && !p->state_based && !s && !W && sizeof(T) == (p->prob.fp64 ? 8 : 4);
    if (!aff) return force_plain<T>(p, u, s, L, W, st);
    if (p->dim == 2) return force_bond_pipeline<T, 2, false>(p, u, s, nullptr, nullptr, L, W, st, true);
    return force_bond_pipeline<T, 3, false>(p, u, s, nullptr, nullptr, L, W, st, true);
}

// Instantiated once: the pipelines of each precision and dimension in
// pd_force_f32_2d.cu, pd_force_f32_3d.cu, pd_force_f64_2d.cu and
// pd_force_f64_3d.cu, the dispatch with the 3D ones.
#define PD_FORCE_PIPELINES(EXTERN, T, D)                                                                          \
    EXTERN template pd_status force_bond_pipeline<T, D, false>(pd_plan *, const T *, const T *, const uint8_t *,   \
                                                               const T *, T *, T *, cudaStream_t, bool);           \
    EXTERN template pd_status force_bond_pipeline<T, D, true>(pd_plan *, const T *, const T *, const uint8_t *,    \
                                                              const T *, T *, T *, cudaStream_t, bool);            \
    EXTERN template pd_status launch_comb<T, CombForce<T, D, false>>(pd_plan *, const CombForce<T, D, false> &,    \
                                                                     cudaStream_t);
#define PD_FORCE_DISPATCH(EXTERN, T)                                                                              \
    EXTERN template pd_status weight_gfield<T>(pd_plan *, const T *, const uint8_t *, T *, cudaStream_t);          \
    EXTERN template pd_status force_any<T>(pd_plan *, const T *, const T *, const uint8_t *, const T *, T *, T *,  \
                                           cudaStream_t);                                                          \
    EXTERN template pd_status force_plain<T>(pd_plan *, const T *, const T *, T *, T *, cudaStream_t);             \
    EXTERN template pd_status force_public<T>(pd_plan *, const T *, const T *, T *, T *, cudaStream_t);
#ifndef PD_FORCE_UNIT
#define PD_FORCE_UNIT 0
#endif
#if PD_FORCE_UNIT != 322
PD_FORCE_PIPELINES(extern, float, 2)
#endif
#if PD_FORCE_UNIT != 323
PD_FORCE_PIPELINES(extern, float, 3)
PD_FORCE_DISPATCH(extern, float)
#endif
#if PD_FORCE_UNIT != 642
PD_FORCE_PIPELINES(extern, double, 2)
#endif
#if PD_FORCE_UNIT != 643
PD_FORCE_PIPELINES(extern, double, 3)
PD_FORCE_DISPATCH(extern, double)
#endif

}  // namespace pd


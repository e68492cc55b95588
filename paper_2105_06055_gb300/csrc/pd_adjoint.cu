// pd_force_adjoint: reverse-mode derivative of the weighted bond force.
//
// The paper has no adjoint. Differentiating the quadrature of Eq. 17-18, 75 with
// bond factor v v' (v = chi s) against a cotangent p = dJ/dL gives
//   gu_i = (dL/du)^T p = v [ conv_M(v p)_i - G_ij p_j ]          (the operator is symmetric)
//   gs   = chi { p . conv_M(v u) - p.G.u - Σ_ij conv_M(v p_i u_j)_ij + u . conv_M(v p) }
// (conv_M = FFT convolution with M^ = (K^(k) - K^(0))/N, G = conv_M(v); the P
// terms of C* = conv_M + P cancel exactly). All of it is one fused pass:
//   rows  : FFT_x1 of v u_j (d), v p_j (d), v (p_i u_j + p_j u_i)/2 (d(d+1)/2)
//   cols  : FFT_x2 (3D)
//   last  : FFT, Y1 = M^ (v u), Y2 = M^ (v p), T3 = Σ_ij M^_ij (v p_i u_j), inverse
//   cols  : inverse FFT_x2 (3D)
//   rows  : inverse FFT_x1, gu and gs at each node.
#include "pd_ops.cuh"

namespace pd {

template <typename T>
pd_status weight_gfield(pd_plan *p, const T *s, const uint8_t *lam, T *G, cudaStream_t st);

namespace {

// Two consecutive values of a caller's field, which may start on any element:
// one vector access when it starts on a pair's boundary.
template <typename T>
__device__ __forceinline__ void load_two(bool pairs, const T *p, T &a, T &b)
{
    if (pairs) {
        load_pair(p, a, b);
    } else {
        a = p[0];
        b = p[1];
    }
}
template <typename T>
__device__ __forceinline__ void store_two(bool pairs, T *p, T a, T b)
{
    if (pairs) {
        store2(p, a, b);
    } else {
        p[0] = a;
        p[1] = b;
    }
}

template <typename T, int D>
struct ProAdj {
    static constexpr int NC = Sym<D>::n;
    static constexpr int kFin = 0, kFout = 2 * D + NC, kNB = 0, kDim = D;
    const T *u, *pv, *s;
    bool pairs;  // they start on pair boundaries
    const uint8_t *chi;
    int64_t N;
    int n1;
    cx<T> *spec;
    int64_t fstride;
    __device__ const cx<T> *spec_in(int) const { return nullptr; }
    __device__ cx<T> *spec_out(int f) const { return spec + f * fstride; }
    __device__ const uint8_t *nb_src(int) const { return nullptr; }
    __device__ void block_done(DSum &) const {}
    struct Nd {
        T ua[D], ub[D], pa[D], pb[D], sa, sb;
        uchar2 in;
    };
    __device__ __forceinline__ void load(Nd &nd, int64_t p0, int o) const
    {
        nd.in = *reinterpret_cast<const uchar2 *>(chi + p0 + o);
        nd.sa = nd.sb = T(1);
        if (s) load_two(pairs, s + p0 + o, nd.sa, nd.sb);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            load_two(pairs, u + (j * N + p0) + o, nd.ua[j], nd.ub[j]);
            load_two(pairs, pv + (j * N + p0) + o, nd.pa[j], nd.pb[j]);
        }
    }
    __device__ __forceinline__ void node2(const RowCtx &, int, Nd &nd, const T *, const T *, T *o0, T *o1,
                                          DSum &) const
    {
        node(nd.in.x ? nd.sa : T(0) * nd.sa, nd.ua, nd.pa, o0);
        node(nd.in.y ? nd.sb : T(0) * nd.sb, nd.ub, nd.pb, o1);
    }
    __device__ __forceinline__ void node(T v, const T *uu, const T *pp, T *out) const
    {
#pragma unroll
        for (int j = 0; j < D; ++j) {
            out[j] = v * uu[j];
            out[D + j] = v * pp[j];
        }
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int a = Sym<D>::i(c), b = Sym<D>::j(c);
            out[2 * D + c] = v * T(0.5) * (pp[a] * uu[b] + pp[b] * uu[a]);
        }
    }
};

template <typename T, int D>
struct CombAdj {
    static constexpr int NC = Sym<D>::n;
    static constexpr int kFin = 2 * D + NC, kFout = 2 * D + 1, kTab = NC, kDim = D;
    Model<T> m;
    __device__ int slot_in(int f) const { return f; }
    __device__ int slot_out(int f) const { return f; }
    __device__ const T *table(int c) const { return m.mhat + c * m.fold_sz; }
    __device__ __forceinline__ void combine(const T *t, bool fy, bool fz, const cx<T> *in, cx<T> *out) const
    {
        T M[9];
        load_mhat_s(D, t, fy, fz, M);
        mat_vec<T, D>(M, in, out);
        mat_vec<T, D>(M, in + D, out + D);
        cx<T> acc = mk(T(0), T(0));
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const int a = Sym<D>::i(c), b = Sym<D>::j(c);
            const T w = (a == b) ? M[3 * a + b] : T(2) * M[3 * a + b];
            acc = acc + scale(in[2 * D + c], w);
        }
        out[2 * D] = acc;
    }
};

template <typename T, int D>
struct EpiAdj {
    static constexpr int NC = Sym<D>::n;
    static constexpr int kFin = 2 * D + 1, kFout = 0, kNB = 0, kDim = D;
    const T *u, *pv, *s, *G;
    const uint8_t *chi;
    T *gu, *gs;
    bool pairs;  // u, pv, s, gu and gs start on pair boundaries
    int64_t N;
    int n1;
    const cx<T> *spec;
    int64_t fstride;
    __device__ const cx<T> *spec_in(int f) const { return spec + f * fstride; }
    __device__ cx<T> *spec_out(int) const { return nullptr; }
    __device__ const uint8_t *nb_src(int) const { return nullptr; }
    __device__ void block_done(DSum &) const {}
    struct Nd {
        T ua[D], ub[D], pa[D], pb[D], ga[NC], gb[NC], sa, sb;
        uchar2 in;
    };
    __device__ __forceinline__ void load(Nd &nd, int64_t p0, int o) const
    {
        nd.in = *reinterpret_cast<const uchar2 *>(chi + p0 + o);
        nd.sa = nd.sb = T(1);
        if (s) load_two(pairs, s + p0 + o, nd.sa, nd.sb);
#pragma unroll
        for (int j = 0; j < D; ++j) {
            load_two(pairs, u + (j * N + p0) + o, nd.ua[j], nd.ub[j]);
            load_two(pairs, pv + (j * N + p0) + o, nd.pa[j], nd.pb[j]);
        }
#pragma unroll
        for (int k = 0; k < NC; ++k) load_pair(G + (k * N + p0) + o, nd.ga[k], nd.gb[k]);
    }
    __device__ __forceinline__ void node2(const RowCtx &c, int o, Nd &nd, const T *in0, const T *in1, T *, T *,
                                          DSum &) const
    {
        T xa[D], xb[D], ya, yb;
        node(nd.in.x != 0, nd.in.x ? nd.sa : T(0) * nd.sa, nd.ua, nd.pa, nd.ga, in0, xa, ya);
        node(nd.in.y != 0, nd.in.y ? nd.sb : T(0) * nd.sb, nd.ub, nd.pb, nd.gb, in1, xb, yb);
        if (gu) {
#pragma unroll
            for (int i = 0; i < D; ++i) store_two(pairs, gu + (i * N + c.p0) + o, xa[i], xb[i]);
        }
        if (gs) store_two(pairs, gs + c.p0 + o, ya, yb);
    }
    __device__ __forceinline__ void node(bool inb, T v, const T *uu, const T *pp, const T *g, const T *in, T *x,
                                         T &y) const
    {
        T Gu[D], Gp[D];
#pragma unroll
        for (int j = 0; j < D; ++j) Gu[j] = Gp[j] = T(0);
        if (inb) {
            sym_apply<T, D>(g, uu, Gu);
            sym_apply<T, D>(g, pp, Gp);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) x[i] = v * (in[D + i] - Gp[i]);
        T acc = -in[2 * D];
#pragma unroll
        for (int i = 0; i < D; ++i) acc += pp[i] * in[i] - pp[i] * Gu[i] + uu[i] * in[D + i];
        y = inb ? acc : T(0);
    }
};

template <typename T, int D>
pd_status adjoint_pipeline(pd_plan *p, const T *u, const T *s, const T *pv, const T *G, T *gu, T *gs,
                           cudaStream_t st)
{
    cx<T> *spec = reinterpret_cast<cx<T> *>(spec_buf<T>(p));
    const int64_t fs = p->N / 2;
    constexpr int FI = 2 * D + Sym<D>::n, FO = 2 * D + 1;
    PD_TRY(check_slots<T>(p, FI));
    const uintptr_t any = (uintptr_t)u | (uintptr_t)pv | (uintptr_t)s | (uintptr_t)gu | (uintptr_t)gs;
    const bool pairs = any % (2 * sizeof(T)) == 0;
    ProAdj<T, D> pro{u, pv, s, pairs, p->chi, p->N, p->n1, spec, fs};
    PD_TRY(launch_rows<T>(p, pro, st));
    if (D == 3) PD_TRY(col_pass<T>(p, 0, FI, false, st));
    CombAdj<T, D> cmb{model_view<T>(p)};
    PD_TRY(launch_comb<T>(p, cmb, st));
    if (D == 3) PD_TRY(col_pass<T>(p, 0, FO, true, st));
    EpiAdj<T, D> epi{u, pv, s, G, p->chi, gu, gs, pairs, p->N, p->n1, spec, fs};
    PD_TRY(launch_rows<T>(p, epi, st));
    return PD_OK;
}

template <typename T>
pd_status adjoint_any(pd_plan *p, const T *u, const T *s, const T *pv, T *gu, T *gs, cudaStream_t st)
{
    const T *G = sizeof(T) == 8 ? (const T *)p->G64 : (const T *)p->G32;
    if (s) {
        PD_TRY(weight_gfield<T>(p, s, nullptr, (T *)p->Gw, st));
        G = (const T *)p->Gw;
    }
    if (p->dim == 2) return adjoint_pipeline<T, 2>(p, u, s, pv, G, gu, gs, st);
    return adjoint_pipeline<T, 3>(p, u, s, pv, G, gu, gs, st);
}

}  // namespace

// The adjoint passes for node weight s with its boundary field G given (the
// dynamic adjoint keeps G current as the integrity index changes).
template <typename T>
pd_status adjoint_weighted(pd_plan *p, const T *u, const T *s, const T *pv, const T *G, T *gu, T *gs,
                           cudaStream_t st)
{
    if (p->dim == 2) return adjoint_pipeline<T, 2>(p, u, s, pv, G, gu, gs, st);
    return adjoint_pipeline<T, 3>(p, u, s, pv, G, gu, gs, st);
}
template pd_status adjoint_weighted<float>(pd_plan *, const float *, const float *, const float *, const float *,
                                           float *, float *, cudaStream_t);
template pd_status adjoint_weighted<double>(pd_plan *, const double *, const double *, const double *,
                                            const double *, double *, double *, cudaStream_t);

}  // namespace pd

using namespace pd;

extern "C" pd_status pd_force_adjoint(pd_plan *p, const void *u, const void *s, const void *gL, void *gu, void *gs,
                                      void *stream)
{
    if (!p || !u || !gL) {
        set_error("pd_force_adjoint: null plan, u or gL");
        return PD_ERR_ARG;
    }
    if (p->state_based || p->nonlinear) {
        set_error("pd_force_adjoint: linearized bond model only");
        return PD_ERR_ARG;
    }
    if (!gu && !gs) return PD_OK;
    cudaStream_t st = (cudaStream_t)stream;
    if (p->prob.fp64)
        return adjoint_any<double>(p, (const double *)u, (const double *)s, (const double *)gL, (double *)gu,
                                   (double *)gs, st);
    return adjoint_any<float>(p, (const float *)u, (const float *)s, (const float *)gL, (float *)gu, (float *)gs, st);
}

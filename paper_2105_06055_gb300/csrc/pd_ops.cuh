// Per-node and per-mode functors of the FCBM-EC operators (private).
//
// Notation: v = chi_B s is the node weight (s = 1, lambda or sqrt(c/c0)),
// conv_M(f) = IFFT(M^ FFT(f)) = C*f dV - P f with M^ = (K^(k) - K^(0))/N
// (Eq. 56-57; the 1/N of the inverse transform is folded into M^), and
// G_ij = conv_M(v)_ij. Then, algebraically identical to Eq. 100-102,
//   L_i = v [ conv_M(v u_j)_i - G_ij u_j ]
//   W   = 1/2 v [ Σ_ij conv_M(v u_i u_j)_ij - 2 u_i conv_M(v u_j)_i + u_i G_ij u_j ]
// (the P terms cancel exactly), which avoids the cancellation between
// C*(v u) and (C*v) u in finite precision. For v = chi_B, G is zero in the
// delta-interior and is kept as a sparse list of boundary nodes, whose G u the
// epilogue subtracts.
#pragma once

#include "pd_affine.cuh"
#include "pd_plan.cuh"

namespace pd {

// component order of symmetric tensors
template <int D>
struct Sym;
template <>
struct Sym<2> {
    static constexpr int n = 3;
    __host__ __device__ static constexpr int i(int c) { return c == 0 ? 0 : c == 1 ? 1 : 0; }
    __host__ __device__ static constexpr int j(int c) { return c == 0 ? 0 : c == 1 ? 1 : 1; }
};
template <>
struct Sym<3> {
    static constexpr int n = 6;
    __host__ __device__ static constexpr int i(int c) { return c < 3 ? c : (c == 5 ? 1 : 0); }
    __host__ __device__ static constexpr int j(int c) { return c < 3 ? c : (c == 3 ? 1 : 2); }
};

template <typename T, int D>
__device__ __forceinline__ void mat_vec(const T *M, const cx<T> *x, cx<T> *y)
{
#pragma unroll
    for (int i = 0; i < D; ++i) {
        cx<T> acc = mk(T(0), T(0));
#pragma unroll
        for (int j = 0; j < D; ++j) acc = acc + scale(x[j], M[3 * i + j]);
        y[i] = acc;
    }
}

// y_i += G_ij x_j for a symmetric tensor stored in Sym order
template <typename T, int D>
__device__ __forceinline__ void sym_apply(const T *g, const T *x, T *y)
{
#pragma unroll
    for (int c = 0; c < Sym<D>::n; ++c) {
        const int a = Sym<D>::i(c), b = Sym<D>::j(c);
        y[a] += g[c] * x[b];
        if (a != b) y[b] += g[c] * x[a];
    }
}

template <typename T>
struct vec2;
template <>
struct vec2<float> {
    using type = float2;
};
template <>
struct vec2<double> {
    using type = double2;
};
template <typename T>
__device__ __forceinline__ typename vec2<T>::type load2(const T *p)
{
    return *reinterpret_cast<const typename vec2<T>::type *>(p);
}

template <typename T>
__device__ __forceinline__ void store2(T *p, T a, T b)
{
    typename vec2<T>::type v;
    v.x = a;
    v.y = b;
    *reinterpret_cast<typename vec2<T>::type *>(p) = v;
}

template <typename T>
__device__ __forceinline__ void load_pair(const T *p, T &a, T &b)
{
    const typename vec2<T>::type v = load2(p);
    a = v.x;
    b = v.y;
}

// masks of the nodes o, o + 1 of the tile from staged byte field 0: chi is its
// low bit
template <typename T>
__device__ __forceinline__ void chi_pair(const RowCtx &c, int o, T &va, T &vb)
{
    const uchar2 b = c.b2(0, o);
    va = (b.x & 1) ? T(1) : T(0);
    vb = (b.y & 1) ? T(1) : T(0);
}

// Node weight next to chi: s (a positive field) or lambda (bytes), or neither.
template <typename T>
struct NodeWeight {
    const T *s;
    const uint8_t *lam;
    __device__ __forceinline__ void load(int64_t p, T &a, T &b) const
    {
        a = b = T(1);
        if (s) load_pair(s + p, a, b);
        if (lam) {
            const uchar2 l = *reinterpret_cast<const uchar2 *>(lam + p);
            a = l.x ? T(1) : T(0);
            b = l.y ? T(1) : T(0);
        }
    }
};

// ---------------------------------------------------------------------------
// Forward prologue: fields v u_j (D) [and v u_i u_j (ncomp) when ENERGY]
// ---------------------------------------------------------------------------
// with an affine view, u - a is transformed instead of u (pd_affine.cuh)
template <typename T, int D, bool ENERGY>
struct ProForce {
    static constexpr int kFin = 0, kFout = D + (ENERGY ? Sym<D>::n : 0), kNB = 1, kDim = D;
    const T *u;
    NodeWeight<T> w;
    const uint8_t *chi;
    int64_t N;
    int n1;
    cx<T> *spec;
    int64_t fstride;
    AffineView<T> aff;  // coef null: none
    __device__ const cx<T> *spec_in(int) const { return nullptr; }
    __device__ cx<T> *spec_out(int f) const { return spec + f * fstride; }
    __device__ const uint8_t *nb_src(int) const { return chi; }
    __device__ __forceinline__ void node1(T v, const T *uu, T *out) const
    {
#pragma unroll
        for (int j = 0; j < D; ++j) out[j] = v * uu[j];
        if constexpr (ENERGY) {
#pragma unroll
            for (int q = 0; q < Sym<D>::n; ++q) out[D + q] = v * uu[Sym<D>::i(q)] * uu[Sym<D>::j(q)];
        }
    }
    struct Nd {
        T a[D], b[D], sa, sb;
    };
    __device__ __forceinline__ void load(Nd &nd, int64_t p0, int o) const
    {
#pragma unroll
        for (int j = 0; j < D; ++j) load_pair(u + (j * N + p0) + o, nd.a[j], nd.b[j]);
        w.load(p0 + o, nd.sa, nd.sb);
    }
    __device__ __forceinline__ void node2(const RowCtx &c, int o, Nd &nd, const T *, const T *, T *o0, T *o1,
                                          DSum &) const
    {
        T va, vb;
        chi_pair(c, o, va, vb);
        if (aff.coef) {
            T a[D], b[D];
            const int i1 = o & (n1 - 1);
            const int64_t row = c.row0 + (o >> aff.lg1);
            aff.at(i1, row, D, a);
            aff.at(i1 + 1, row, D, b);
#pragma unroll
            for (int j = 0; j < D; ++j) {
                nd.a[j] -= a[j];
                nd.b[j] -= b[j];
            }
        }
        node1(va * nd.sa, nd.a, o0);
        node1(vb * nd.sb, nd.b, o1);
    }
    __device__ void block_done(DSum &) const {}
};

// ---------------------------------------------------------------------------
// Spectral combine: Y_i = M^_ij X_j [, T = Σ_ij M^_ij Q_ij]
// ---------------------------------------------------------------------------
template <typename T, int D, bool ENERGY>
struct CombForce {
    static constexpr int kFin = D + (ENERGY ? Sym<D>::n : 0);
    static constexpr int kFout = D + (ENERGY ? 1 : 0);
    static constexpr int kTab = Sym<D>::n, kDim = D;
    Model<T> m;
    __device__ int slot_in(int f) const { return f; }
    __device__ int slot_out(int f) const { return f; }
    __device__ const T *table(int c) const { return m.mhat + c * m.fold_sz; }
    __device__ __forceinline__ void combine(const T *t, bool fy, bool fz, const cx<T> *in, cx<T> *out) const
    {
        T M[9];
        load_mhat_s(D, t, fy, fz, M);
        mat_vec<T, D>(M, in, out);
        if constexpr (ENERGY) {
            cx<T> acc = mk(T(0), T(0));
#pragma unroll
            for (int c = 0; c < Sym<D>::n; ++c) {
                const int a = Sym<D>::i(c), b = Sym<D>::j(c);
                const T w = (a == b) ? M[3 * a + b] : T(2) * M[3 * a + b];
                acc = acc + scale(in[D + c], w);
            }
            out[D] = acc;
        }
    }
};

// ---------------------------------------------------------------------------
// Inverse epilogue, plan weight (v = chi_B): sparse boundary field
//   L_i = chi (y_i - G_ij u_j), W = 1/2 chi (y_T - 2 u.y + u.G.u) with G from
//   the boundary list
// ---------------------------------------------------------------------------
// with an affine view the transforms saw u - a; G applies to u - a and the exact
// L(a) is added from the boundary entry's moment row (plain force only)
template <typename T, int D, bool ENERGY>
struct EpiForceSparse {
    static constexpr int kFin = D + (ENERGY ? 1 : 0), kFout = 0, kNB = 1, kDim = D;
    static constexpr bool kEntries = true;
    const T *u;
    const uint8_t *chi;
    const GEntry<T> *gent;
    const int *goff;
    T *L;
    T *W;
    int64_t N;
    int n1;
    const cx<T> *spec;
    int64_t fstride;
    AffineView<T> aff;  // coef null: none
    const T *atab;  // [entries][Sym<D>::n * D]
    __device__ const cx<T> *spec_in(int f) const { return spec + f * fstride; }
    __device__ cx<T> *spec_out(int) const { return nullptr; }
    __device__ const uint8_t *nb_src(int) const { return chi; }
    __device__ __forceinline__ const int *rows_off() const { return goff; }
    // boundary entry k: what it adds to y_i (and y_T) at its node, where chi = 1
    __device__ __forceinline__ void entry(int k, int64_t &p, T *s) const
    {
        const GEntry<T> e = gent[k];
        p = e.p;
        T uu[D], Gu[D];
#pragma unroll
        for (int j = 0; j < D; ++j) {
            uu[j] = u[j * N + p];
            Gu[j] = T(0);
        }
#pragma unroll
        for (int i = 0; i < D; ++i) s[i] = T(0);
        if (!ENERGY && aff.coef) {
            T a[D];
            const int64_t row = p / n1;
            aff.at((int)(p - row * n1), row, D, a);
#pragma unroll
            for (int j = 0; j < D; ++j) uu[j] -= a[j];
            aff_force<T, D>(aff.coef, atab + (int64_t)k * (Sym<D>::n * D), s);
        }
        sym_apply<T, D>(e.g, uu, Gu);
#pragma unroll
        for (int i = 0; i < D; ++i) s[i] -= Gu[i];
        if constexpr (ENERGY) {
            // W = 1/2 (y_T - 2 u.y + u.G.u) with the corrected y: y_T loses u.G.u
            T ugu = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) ugu += uu[i] * Gu[i];
            s[D] = -ugu;
        }
    }
    struct Nd {
        T a[ENERGY ? D : 1], b[ENERGY ? D : 1];
    };
    __device__ __forceinline__ void load(Nd &nd, int64_t p0, int o) const
    {
        if constexpr (ENERGY) {
#pragma unroll
            for (int i = 0; i < D; ++i) load_pair(u + (i * N + p0) + o, nd.a[i], nd.b[i]);
        }
    }
    __device__ __forceinline__ void node2(const RowCtx &c, int o, Nd &nd, const T *in0, const T *in1, T *, T *,
                                          DSum &) const
    {
        const uchar2 b = c.b2(0, o);
        const T va = b.x ? T(1) : T(0), vb = b.y ? T(1) : T(0);
#pragma unroll
        for (int i = 0; i < D; ++i) store2(L + (i * N + c.p0) + o, va * in0[i], vb * in1[i]);
        if constexpr (ENERGY) {
            T ca = T(0), cb = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                ca += nd.a[i] * in0[i];
                cb += nd.b[i] * in1[i];
            }
            if (W) store2(W + c.p0 + o, T(0.5) * va * (in0[D] - T(2) * ca), T(0.5) * vb * (in1[D] - T(2) * cb));
        }
    }
    __device__ void block_done(DSum &) const {}
};

// ---------------------------------------------------------------------------
// Inverse epilogue, node weight s or lambda: dense boundary field G^v
//   L_i = v (y_i - G_ij u_j), W = 1/2 v (y_T - 2 u.y + u.G.u)
// ---------------------------------------------------------------------------
template <typename T, int D, bool ENERGY>
struct EpiForceDense {
    static constexpr int NC = Sym<D>::n;
    static constexpr int kFin = D + (ENERGY ? 1 : 0), kFout = 0, kNB = 1, kDim = D;
    const T *u;
    NodeWeight<T> w;
    const uint8_t *chi;
    const T *G;  // ncomp x N, for the same weight
    T *L;
    T *W;
    int64_t N;
    int n1;
    const cx<T> *spec;
    int64_t fstride;
    __device__ const cx<T> *spec_in(int f) const { return spec + f * fstride; }
    __device__ cx<T> *spec_out(int) const { return nullptr; }
    __device__ const uint8_t *nb_src(int) const { return chi; }
    __device__ __forceinline__ void node1(T v, const T *uu, const T *gg, const T *in, T *Lo, T &Wo) const
    {
        T g[NC], Gu[D];
#pragma unroll
        for (int j = 0; j < D; ++j) Gu[j] = T(0);
#pragma unroll
        for (int q = 0; q < NC; ++q) g[q] = (v != T(0)) ? gg[q] : T(0);
        sym_apply<T, D>(g, uu, Gu);
#pragma unroll
        for (int i = 0; i < D; ++i) Lo[i] = v * (in[i] - Gu[i]);
        if constexpr (ENERGY) {
            T uc = T(0), ugu = T(0);
#pragma unroll
            for (int i = 0; i < D; ++i) {
                uc += uu[i] * in[i];
                ugu += uu[i] * Gu[i];
            }
            Wo = T(0.5) * v * (in[D] - T(2) * uc + ugu);
        }
    }
    struct Nd {
        T ua[D], ub[D], ga[NC], gb[NC], sa, sb;
    };
    __device__ __forceinline__ void load(Nd &nd, int64_t p0, int o) const
    {
#pragma unroll
        for (int j = 0; j < D; ++j) load_pair(u + (j * N + p0) + o, nd.ua[j], nd.ub[j]);
#pragma unroll
        for (int q = 0; q < NC; ++q) load_pair(G + (q * N + p0) + o, nd.ga[q], nd.gb[q]);
        w.load(p0 + o, nd.sa, nd.sb);
    }
    __device__ __forceinline__ void node2(const RowCtx &c, int o, Nd &nd, const T *in0, const T *in1, T *, T *,
                                          DSum &) const
    {
        T va, vb;
        chi_pair(c, o, va, vb);
        va *= nd.sa;
        vb *= nd.sb;
        T a[D], b[D], wa = T(0), wb = T(0);
        node1(va, nd.ua, nd.ga, in0, a, wa);
        node1(vb, nd.ub, nd.gb, in1, b, wb);
#pragma unroll
        for (int i = 0; i < D; ++i) store2(L + (i * N + c.p0) + o, a[i], b[i]);
        if constexpr (ENERGY) {
            if (W) store2(W + c.p0 + o, wa, wb);
        }
    }
    __device__ void block_done(DSum &) const {}
};

}  // namespace pd

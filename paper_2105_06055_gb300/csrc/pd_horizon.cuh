// Direct horizon sums on shared-memory tiles (private): the boundary field of
// a node weight and the Eq. 47 energy density.
//
// Both sums read every node's horizon neighbourhood (a few dozen to a few
// hundred nodes). A block takes a tile of nodes with its halo into shared
// memory once (periodic wrap and masks applied there), keeps the bond table
// beside it in the plan's precision, and each thread sums kNodes nodes, so a
// bond's coefficients are fetched once per kNodes nodes and the inner loop is
// shared-memory loads and FMAs only. The kernels that read the neighbours and
// the FP64 bond table from global memory for every node and bond (k_gfield
// below and the energy kernel's counterpart) are bound by the FP64
// conversions of the table (the GB300 converts and multiplies FP64 at 1/64 of
// its FP32 rate) and by the address arithmetic; they remain for horizons that reach
// more than kHzReach cells along the last axis, the most the column loops are unrolled
// for, or whose tile does not fit in shared memory. The step is steep: on a 1024 x 512
// plate in FP32 a weighted force takes 33 us at a reach of 4 cells and 235 at 5, a
// fracture step with the energy sum 53 and 132.
#pragma once

#include <limits>

#include "pd_ops.cuh"
#include "pd_plan.cuh"

namespace pd {

constexpr int kHzX = 32, kHzY = 8, kNodes = 4;  // threads per block 32 x 8, nodes per thread
constexpr size_t kHzSmem = 100 * 1024;          // two blocks per SM at least

// Tile geometry: 3D 32 x 8 x 4 nodes, 2D 32 x 32; a thread's kNodes nodes follow
// each other along the tile's last axis (x3 in 3D, x2 in 2D).
struct HzTile {
    int n1, n2, n3;
    int r1, r2, r3;    // halo
    int p, rows, nz;   // halo tile: pitch (x1), rows (x2), planes (x3)
    int step;          // tile elements between a thread's nodes (along the last axis)
    int two;           // 2D
    int rb, rc;        // reach across (x2 in 3D, 0 in 2D) and along the last axis
    int ncol;          // columns of the horizon's box: offsets (o1, ob), all oc
};

inline HzTile hz_tile(int dim, int n1, int n2, int n3, const HorizonDev &hz)
{
    HzTile t;
    t.n1 = n1;
    t.n2 = n2;
    t.n3 = n3;
    t.r1 = hz.r[0];
    t.r2 = hz.r[1];
    t.r3 = dim == 3 ? hz.r[2] : 0;
    t.two = dim == 2;
    t.p = kHzX + 2 * t.r1;
    t.rows = (t.two ? kHzY * kNodes : kHzY) + 2 * t.r2;
    t.nz = t.two ? 1 : kNodes + 2 * t.r3;
    t.step = t.two ? t.p : t.rows * t.p;
    t.rb = t.two ? 0 : t.r2;
    t.rc = t.two ? t.r2 : t.r3;
    t.ncol = (2 * t.r1 + 1) * (2 * t.rb + 1);
    return t;
}

inline dim3 hz_grid(const HzTile &t)
{
    return t.two ? dim3((unsigned)(t.n1 / kHzX), (unsigned)((t.n2 + kHzY * kNodes - 1) / (kHzY * kNodes)))
                 : dim3((unsigned)(t.n1 / kHzX), (unsigned)(t.n2 / kHzY), (unsigned)(t.n3 / kNodes));
}

// Calls fill(tile element, node) for the halo tile of this block (all threads).
template <class Fill>
__device__ __forceinline__ void hz_fill(const HzTile &t, Fill fill)
{
    const int x0 = blockIdx.x * kHzX - t.r1, y0 = blockIdx.y * (t.two ? kHzY * kNodes : kHzY) - t.r2;
    const int z0 = t.two ? 0 : (int)blockIdx.z * kNodes - t.r3;
    // one warp per row of the tile, two columns per lane (more past 64);
    // (y, z) run along without divisions
    const int lane = threadIdx.x;
    int yr = threadIdx.y, zr = 0;
    while (yr >= t.rows) {
        yr -= t.rows;
        ++zr;
    }
    const bool rest = lane + 32 < t.p;
    const int xa = (x0 + lane) & (t.n1 - 1), xb = (x0 + lane + 32) & (t.n1 - 1);
#pragma unroll 4
    while (zr < t.nz) {
        const int y = (y0 + yr) & (t.n2 - 1), z = t.two ? 0 : (z0 + zr) & (t.n3 - 1);
        const int64_t row = ((int64_t)z * t.n2 + y) * t.n1;
        const int e = (zr * t.rows + yr) * t.p + lane;
        fill(e, row + xa);
        if (rest) fill(e + 32, row + xb);
        yr += kHzY;
        while (yr >= t.rows) {
            yr -= t.rows;
            ++zr;
        }
    }
    if (t.p > 64)  // reach above 16 cells (uneven spacings)
        for (int r = threadIdx.y; r < t.rows * t.nz; r += kHzY) {
            const int y = (y0 + r % t.rows) & (t.n2 - 1), z = t.two ? 0 : (z0 + r / t.rows) & (t.n3 - 1);
            const int64_t row = ((int64_t)z * t.n2 + y) * t.n1;
            for (int x = lane + 64; x < t.p; x += 32) fill(r * t.p + x, row + ((x0 + x) & (t.n1 - 1)));
        }
}

// Tile element and node of this thread's node m; false past the grid (2D, n2 < 32).
__device__ __forceinline__ bool hz_node(const HzTile &t, int m, int64_t &node)
{
    const int x = blockIdx.x * kHzX + threadIdx.x;
    const int y = t.two ? ((int)blockIdx.y * kHzY + (int)threadIdx.y) * kNodes + m
                        : (int)blockIdx.y * kHzY + (int)threadIdx.y;
    const int z = t.two ? 0 : (int)blockIdx.z * kNodes + m;
    node = ((int64_t)z * t.n2 + y) * t.n1 + x;
    return y < t.n2;
}
__device__ __forceinline__ int hz_elem0(const HzTile &t)
{
    return ((t.two ? 0 : t.r3) * t.rows + (int)threadIdx.y * (t.two ? kNodes : 1) + t.r2) * t.p +
           (int)threadIdx.x + t.r1;
}
// The horizon as columns along the last axis: column (o1, ob) has its bonds at
// oc = -zmax ... zmax. A thread loads the kNodes + 2 zmax tile values of a column
// once and uses them for all of its nodes and bonds (at delta = 3 in 3D, 210
// shared-memory loads per thread instead of one per node and bond, 488).
// The tables are made once per plan (k_hz_tables): the bond values need FP64
// divisions and conversions, which every block would otherwise repeat.
constexpr int kHzReach = 4;      // largest reach along the last axis the kernels are unrolled for
constexpr int kHzMaxCols = 1024;  // most columns
// slot of (column, oc): col (2 rc + 1) + oc + rc; column (o1, ob):
// (ob + rb) (2 r1 + 1) + o1 + r1
template <typename T>
struct HzTables {
    const T *coef;    // [slots][8 or 4]: C in Sym order, padded
    const T *bond;    // [slots][4]: xi, c / |xi|^2
    const int2 *col;  // {tile offset, first slot} of the columns, ordered by zmax: those of
                      // one half of the horizon (opposite columns), then all
    const int *grp;   // [2][kHzReach + 2]: where each zmax begins in the two lists
};
inline size_t hz_table_values(int dim, const HzTile &t) { return (size_t)((dim == 3 ? 8 : 4) + 4) * t.ncol * (2 * t.rc + 1); }
template <typename T>
inline HzTables<T> hz_tables(const pd_plan *p, const HzTile &t)
{
    const T *v = reinterpret_cast<const T *>(sizeof(T) == 8 ? (const void *)p->hzt64 : (const void *)p->hzt32);
    const size_t slots = (size_t)t.ncol * (2 * t.rc + 1);
    return {v, v + (p->dim == 3 ? 8 : 4) * slots, p->hzcol,
            reinterpret_cast<const int *>(p->hzcol + 2 * t.ncol)};
}
inline size_t hz_col_entries(const HzTile &t) { return 2 * (size_t)t.ncol + kHzReach + 2; }
// (one block; the value arrays are zero before)
template <typename T>
__global__ void k_hz_tables(HzTile t, HorizonDev hz, int dim, double dx1, double dx2, double dx3, T *val, int2 *cols)
{
    const int nc = dim == 3 ? 6 : 3, cp = dim == 3 ? 8 : 4, nz = 2 * t.rc + 1;
    T *bond = val + (size_t)cp * t.ncol * nz;
    __shared__ int zmax[kHzMaxCols];
    for (int c = threadIdx.x; c < t.ncol; c += blockDim.x) zmax[c] = -1;
    __syncthreads();
    for (int c = threadIdx.x; c < hz.cnt; c += blockDim.x) {
        const int o1 = hz.off[3 * c], ob = t.two ? 0 : hz.off[3 * c + 1], oc = hz.off[3 * c + (t.two ? 1 : 2)];
        const int col = (ob + t.rb) * (2 * t.r1 + 1) + o1 + t.r1, slot = col * nz + oc + t.rc;
        atomicMax(&zmax[col], oc < 0 ? -oc : oc);
        const double x[3] = {hz.off[3 * c] * dx1, hz.off[3 * c + 1] * dx2, hz.off[3 * c + 2] * dx3};
        double tr = 0.0, r2 = 0.0;
        for (int j = 0; j < dim; ++j) {
            tr += hz.c[j * hz.cnt + c];  // the diagonal components come first
            r2 += x[j] * x[j];
        }
        for (int k = 0; k < nc; ++k) val[cp * slot + k] = (T)hz.c[k * hz.cnt + c];
        for (int j = 0; j < dim; ++j) bond[4 * slot + j] = (T)x[j];
        bond[4 * slot + 3] = (T)(tr / r2);
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    int *grp = reinterpret_cast<int *>(cols + 2 * t.ncol);
    for (int list = 0; list < 2; ++list) {
        int n = 0;
        for (int z = 0; z <= kHzReach; ++z) {
            grp[list * (kHzReach + 2) + z] = n;
            for (int c = 0; c < (list ? t.ncol : t.ncol / 2); ++c)
                if (zmax[c] == z)
                    cols[list * t.ncol + n++] = make_int2(
                        (c / (2 * t.r1 + 1) - t.rb) * t.p + c % (2 * t.r1 + 1) - t.r1, c * nz);
        }
        grp[list * (kHzReach + 2) + kHzReach + 1] = n;
    }
}

__device__ __forceinline__ float weight_value(float s) { return s; }
__device__ __forceinline__ double weight_value(double s) { return s; }
__device__ __forceinline__ float weight_value(uint8_t s) { return s ? 1.f : 0.f; }

// Boundary field of the node weight v = chi s (s null: chi), one thread per
// node, neighbours from global memory; for the horizons that the tile form does not
// take (launch_gfield). A launch with `changed` does nothing while *changed is 0.
//   G_c(x) = Σ_H C_c(xi) dV (v(x+xi) - v(x)),  G = 0 where chi = 0
// (Eq. 100 with the difference kernel; for v = chi this is
// -(Σ_H C dV (1 - chi(x+xi))), zero in the delta-interior).
template <typename T, typename V, typename Acc>
__global__ void k_gfield(int n1, int n2, int n3, HorizonDev hz, int ncomp, const uint8_t *chi,
                         const V *s, T *G, int64_t N, const int *changed)
{
    if (changed && !*changed) return;
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= N) return;
    int i1, i2, i3;
    node_coords(p, n1, n2, i1, i2, i3);
    Acc acc[6] = {0, 0, 0, 0, 0, 0};
    if (chi[p]) {
        const Acc vp = s ? (Acc)weight_value(s[p]) : Acc(1);
        for (int c = 0; c < hz.cnt; ++c) {
            const int a = (i1 + hz.off[3 * c]) & (n1 - 1);
            const int b = (i2 + hz.off[3 * c + 1]) & (n2 - 1);
            const int e = (i3 + hz.off[3 * c + 2]) & (n3 - 1);
            const int64_t q = ((int64_t)e * n2 + b) * n1 + a;
            const Acc vq = chi[q] ? (s ? (Acc)weight_value(s[q]) : Acc(1)) : Acc(0);
            const Acc dv = vq - vp;
            if (dv != Acc(0))
                for (int k = 0; k < ncomp; ++k) acc[k] += (Acc)hz.c[k * hz.cnt + c] * dv;
        }
    }
    for (int k = 0; k < ncomp; ++k) G[k * N + p] = (T)acc[k];
}

// One pair of opposite columns: the bonds (o, oc) of column `col` and their
// opposites; C is even, so each pair adds C_c ((v(x+xi) - v(x)) + (v(x-xi) - v(x))).
// CENTER: the column of x itself, opposite bonds oc and -oc.
template <typename T, int NC, int CP, int Z, bool CENTER>
__device__ __forceinline__ void gfield_column(const T *tile, const T *coef, int e, int d, int step, int rc,
                                              const T *v, T (&acc)[kNodes][NC])
{
    T a[kNodes + 2 * Z], b[kNodes + 2 * Z];
#pragma unroll
    for (int z = 0; z < kNodes + 2 * Z; ++z) {
        a[z] = tile[e + d + (z - Z) * step];
        b[z] = CENTER ? a[z] : tile[e - d + (z - Z) * step];
    }
#pragma unroll
    for (int oc = CENTER ? 1 : -Z; oc <= Z; ++oc) {
        T w[NC];
#pragma unroll
        for (int k = 0; k < NC; k += 2) {  // CP is even, the table on a 16-byte boundary
            const typename vec2<T>::type c2 = *reinterpret_cast<const typename vec2<T>::type *>(coef + CP * (rc + oc) + k);
            w[k] = c2.x;
            if (k + 1 < NC) w[k + 1] = c2.y;
        }
#pragma unroll
        for (int m = 0; m < kNodes; ++m) {
            const T dv = (a[m + Z + oc] - v[m]) + (b[m + Z - oc] - v[m]);
#pragma unroll
            for (int k = 0; k < NC; ++k) acc[m][k] += w[k] * dv;
        }
    }
}

// The same field on tiles, column by column. Bound by instruction issue (the sums
// are half of its instructions, the rest loads and the fill of the halo tile) and,
// below four blocks an SM, by the latency of the fill: 111 us at 128^3 and 122 bonds
// with 80 registers and rows filled two at a time, 97 with 64 registers and four.
// 8 nodes per thread issue 12% fewer instructions but need 128 registers: 113 us.
template <typename T, typename V, int NC>
__global__ void __launch_bounds__(kHzX *kHzY, sizeof(T) == 4 ? 4 : 1) k_gfield_tile(HzTile t, HzTables<T> tab,
                                                           const uint8_t *__restrict__ chi,
                                                           const V *__restrict__ s, T *__restrict__ G, int64_t N,
                                                           const int *changed)
{
    if (changed && !*changed) return;
    constexpr int CP = NC == 6 ? 8 : 4;  // coefficients per bond, padded to whole vectors
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T *coef = reinterpret_cast<T *>(sm_raw);
    const int nz = 2 * t.rc + 1, slots = t.ncol * nz;
    int2 *col = reinterpret_cast<int2 *>(coef + (size_t)CP * slots);
    T *tile = reinterpret_cast<T *>(col + ((t.ncol / 2 + 1) & ~1));
    const int tid = threadIdx.y * kHzX + threadIdx.x;
    for (int c = tid; c < t.ncol / 2; c += kHzX * kHzY) col[c] = tab.col[c];
    for (int c = tid; c < CP * slots / 4; c += kHzX * kHzY) {
#pragma unroll
        for (int k = 0; k < 4; ++k) coef[4 * c + k] = tab.coef[4 * c + k];
    }
    T lo = std::numeric_limits<T>::infinity(), hi = -lo;  // range of the weights this thread loads
    bool nan = false;
    hz_fill(t, [&](int e, int64_t q) {
        const uint8_t in = chi[q];
        const T w = s ? (T)weight_value(s[q]) : T(1);
        const T x = in ? w : T(0);
        lo = x < lo ? x : lo;
        hi = x > hi ? x : hi;
        nan = nan || x != x;
        tile[e] = x;
    });
    __syncthreads();
    // the field is 0 where the weight does not change: the inside of a body with
    // weight 1 (a plan's own field in FP64 would otherwise cost more than the
    // per-node sum, which skips equal weights)
    const bool flat = __syncthreads_and(!nan && (lo > hi || (lo == tile[0] && hi == tile[0])));
    const int e0 = hz_elem0(t);
    T v[kNodes], acc[kNodes][NC];
#pragma unroll
    for (int m = 0; m < kNodes; ++m) {
        v[m] = tile[e0 + m * t.step];
#pragma unroll
        for (int k = 0; k < NC; ++k) acc[m][k] = T(0);
    }
    if (!flat) {
        // one loop per zmax: a switch per column cost as many register moves as
        // the sums themselves (118 us at 128^3, 122 bonds)
#define PD_GFIELD_COLUMNS(Z)                                                                                    \
    _Pragma("unroll 1") for (int c = __ldg(tab.grp + Z); c < __ldg(tab.grp + Z + 1); ++c)                        \
    {                                                                                                           \
        const int2 k = col[c];                                                                                  \
        gfield_column<T, NC, CP, Z, false>(tile, coef + CP * k.y, e0, k.x, t.step, t.rc, v, acc);               \
    }
        PD_GFIELD_COLUMNS(0)
        PD_GFIELD_COLUMNS(1)
        PD_GFIELD_COLUMNS(2)
        PD_GFIELD_COLUMNS(3)
        PD_GFIELD_COLUMNS(4)
#undef PD_GFIELD_COLUMNS
        const T *w = coef + (size_t)CP * (t.ncol / 2) * nz;
        switch (t.rc) {  // the column of the node itself reaches as far as any
            case 1: gfield_column<T, NC, CP, 1, true>(tile, w, e0, 0, t.step, t.rc, v, acc); break;
            case 2: gfield_column<T, NC, CP, 2, true>(tile, w, e0, 0, t.step, t.rc, v, acc); break;
            case 3: gfield_column<T, NC, CP, 3, true>(tile, w, e0, 0, t.step, t.rc, v, acc); break;
            case 4: gfield_column<T, NC, CP, 4, true>(tile, w, e0, 0, t.step, t.rc, v, acc); break;
            default: break;
        }
    }
#pragma unroll
    for (int m = 0; m < kNodes; ++m) {
        int64_t p;
        if (!hz_node(t, m, p)) continue;
        const bool in = chi[p] != 0;
#pragma unroll
        for (int k = 0; k < NC; ++k) G[k * N + p] = in ? acc[m][k] : T(0);
    }
}

// Enqueues the boundary field of the weight chi s into G. Tiles for horizons
// that reach at most kHzReach cells along the last axis and whose tile fits.
template <typename T, typename V>
pd_status launch_gfield(const pd_plan *p, const V *s, T *G, const int *changed, cudaStream_t st)
{
    const HzTile t = hz_tile(p->dim, p->n1, p->n2, p->n3, p->hdev);
    const size_t smem = ((size_t)(p->dim == 3 ? 8 : 4) * t.ncol * (2 * t.rc + 1) + (size_t)t.p * t.rows * t.nz) *
                            sizeof(T) +
                        (size_t)((t.ncol / 2 + 1) & ~1) * sizeof(int2);
    if (smem > kHzSmem || t.rc > kHzReach || !p->hzcol) {
        k_gfield<T, V, T><<<(unsigned)((p->N + 127) / 128), 128, 0, st>>>(p->n1, p->n2, p->n3, p->hdev, p->ncomp,
                                                                         p->chi, s, G, p->N, changed);
        PD_LAUNCH_CHECK();
        return PD_OK;
    }
    const auto kern = p->dim == 3 ? k_gfield_tile<T, V, 6> : k_gfield_tile<T, V, 3>;
    PD_TRY(set_smem_attr((const void *)kern, smem));
    kern<<<hz_grid(t), dim3(kHzX, kHzY), smem, st>>>(t, hz_tables<T>(p, t), p->chi, s, G, p->N, changed);
    PD_LAUNCH_CHECK();
    return PD_OK;
}

// Instantiated once, in pd_horizon.cu.
#define PD_GFIELD_INSTANCES(EXTERN)                                                                              \
    EXTERN template pd_status launch_gfield<float, float>(const pd_plan *, const float *, float *, const int *,   \
                                                          cudaStream_t);                                          \
    EXTERN template pd_status launch_gfield<double, double>(const pd_plan *, const double *, double *,            \
                                                            const int *, cudaStream_t);                           \
    EXTERN template pd_status launch_gfield<float, uint8_t>(const pd_plan *, const uint8_t *, float *,            \
                                                            const int *, cudaStream_t);                           \
    EXTERN template pd_status launch_gfield<double, uint8_t>(const pd_plan *, const uint8_t *, double *,          \
                                                             const int *, cudaStream_t);
#ifndef PD_HORIZON_UNIT
PD_GFIELD_INSTANCES(extern)
#endif

}  // namespace pd

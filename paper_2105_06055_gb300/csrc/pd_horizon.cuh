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
// its FP32 rate) and by the address arithmetic; they remain for horizons
// whose tile does not fit.
#pragma once

#include "pd_ops.cuh"
#include "pd_plan.cuh"

namespace pd {

constexpr int kHzX = 32, kHzY = 8, kNodes = 4;  // threads per block 32 x 8, nodes per thread
constexpr size_t kHzSmem = 100 * 1024;          // two blocks per SM at least

// Tile geometry: 3D 32 x 8 x 4 nodes (a thread's nodes along x3), 2D 32 x 32
// (a thread's nodes 8 rows apart along x2).
struct HzTile {
    int n1, n2, n3;
    int r1, r2, r3;    // halo
    int p, rows, nz;   // halo tile: pitch (x1), rows (x2), planes (x3)
    int step;          // tile elements between a thread's nodes
    int two;           // 2D
    int np;            // bond pairs (bonds c and cnt - 1 - c are opposite)
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
    t.step = t.two ? kHzY * t.p : t.rows * t.p;
    t.np = hz.cnt / 2;
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
    const int tid = threadIdx.y * kHzX + threadIdx.x;
    for (int r = tid / 32; r < t.rows * t.nz; r += kHzY) {  // one warp per row of the tile
        const int y = (y0 + r % t.rows) & (t.n2 - 1), z = t.two ? 0 : (z0 + r / t.rows) & (t.n3 - 1);
        const int64_t row = ((int64_t)z * t.n2 + y) * t.n1;
        for (int x = tid % 32; x < t.p; x += 32) fill(r * t.p + x, row + ((x0 + x) & (t.n1 - 1)));
    }
}

// Tile element and node of this thread's node m; false past the grid (2D, n2 < 32).
__device__ __forceinline__ bool hz_node(const HzTile &t, int m, int64_t &node)
{
    const int x = blockIdx.x * kHzX + threadIdx.x;
    const int y = t.two ? (int)blockIdx.y * kHzY * kNodes + (int)threadIdx.y + kHzY * m
                        : (int)blockIdx.y * kHzY + (int)threadIdx.y;
    const int z = t.two ? 0 : (int)blockIdx.z * kNodes + m;
    node = ((int64_t)z * t.n2 + y) * t.n1 + x;
    return y < t.n2;
}
__device__ __forceinline__ int hz_elem0(const HzTile &t)
{
    return ((t.two ? 0 : t.r3) * t.rows + (int)threadIdx.y + t.r2) * t.p + (int)threadIdx.x + t.r1;
}

__device__ __forceinline__ float weight_value(float s) { return s; }
__device__ __forceinline__ double weight_value(double s) { return s; }
__device__ __forceinline__ float weight_value(uint8_t s) { return s ? 1.f : 0.f; }

// Boundary field of the node weight v = chi s (s null: chi), one thread per
// node, neighbours from global memory; for horizons whose tile does not fit in
// shared memory. A launch with `changed` does nothing while *changed is 0.
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

// The same field on tiles: opposite bonds share their coefficients (C is
// even), so a pair adds C_c ((v(x+xi) - v(x)) + (v(x-xi) - v(x))).
template <typename T, typename V, int NC>
__global__ void __launch_bounds__(kHzX *kHzY) k_gfield_tile(HzTile t, HorizonDev hz,
                                                           const uint8_t *__restrict__ chi,
                                                           const V *__restrict__ s, T *__restrict__ G, int64_t N,
                                                           const int *changed)
{
    if (changed && !*changed) return;
    constexpr int CP = NC == 6 ? 8 : 4;  // coefficients per pair, padded to whole vectors
    extern __shared__ __align__(16) unsigned char sm_raw[];
    T *coef = reinterpret_cast<T *>(sm_raw);
    int *off = reinterpret_cast<int *>(coef + (size_t)CP * t.np);
    T *tile = reinterpret_cast<T *>(off + ((t.np + 3) & ~3));
    const int tid = threadIdx.y * kHzX + threadIdx.x;
    for (int c = tid; c < t.np; c += kHzX * kHzY) {
        off[c] = (hz.off[3 * c + 2] * t.rows + hz.off[3 * c + 1]) * t.p + hz.off[3 * c];
#pragma unroll
        for (int k = 0; k < CP; ++k) coef[CP * c + k] = k < NC ? (T)hz.c[k * hz.cnt + c] : T(0);
    }
    hz_fill(t, [&](int e, int64_t q) {
        tile[e] = chi[q] ? (s ? (T)weight_value(s[q]) : T(1)) : T(0);
    });
    __syncthreads();
    const int e0 = hz_elem0(t);
    T v[kNodes], acc[kNodes][NC];
#pragma unroll
    for (int m = 0; m < kNodes; ++m) {
        v[m] = tile[e0 + m * t.step];
#pragma unroll
        for (int k = 0; k < NC; ++k) acc[m][k] = T(0);
    }
#pragma unroll 2
    for (int c = 0; c < t.np; ++c) {
        const int d = off[c];
        T w[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) w[k] = coef[CP * c + k];
#pragma unroll
        for (int m = 0; m < kNodes; ++m) {
            const int e = e0 + m * t.step;
            const T dv = (tile[e + d] - v[m]) + (tile[e - d] - v[m]);
#pragma unroll
            for (int k = 0; k < NC; ++k) acc[m][k] += w[k] * dv;
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

// Enqueues the boundary field of the weight chi s into G.
template <typename T, typename V>
pd_status launch_gfield(const pd_plan *p, const V *s, T *G, const int *changed, cudaStream_t st)
{
    const HzTile t = hz_tile(p->dim, p->n1, p->n2, p->n3, p->hdev);
    const size_t smem = ((size_t)(p->dim == 3 ? 8 : 4) * t.np + (size_t)t.p * t.rows * t.nz) * sizeof(T) +
                        (size_t)((t.np + 3) & ~3) * sizeof(int);
    if (smem > kHzSmem) {
        k_gfield<T, V, T><<<(unsigned)((p->N + 127) / 128), 128, 0, st>>>(p->n1, p->n2, p->n3, p->hdev, p->ncomp,
                                                                         p->chi, s, G, p->N, changed);
        PD_LAUNCH_CHECK();
        return PD_OK;
    }
    const auto kern = p->dim == 3 ? k_gfield_tile<T, V, 6> : k_gfield_tile<T, V, 3>;
    PD_TRY(set_smem_attr((const void *)kern, smem));
    kern<<<hz_grid(t), dim3(kHzX, kHzY), smem, st>>>(t, p->hdev, p->chi, s, G, p->N, changed);
    PD_LAUNCH_CHECK();
    return PD_OK;
}

}  // namespace pd

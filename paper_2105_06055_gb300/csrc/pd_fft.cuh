// Transforms for the FCBM-EC convolutions.
//
// The convolutions of Eq. 57-65 and 95-102 are evaluated with the DFT of
// Eq. 53-54 on the periodic box. A d-dimensional transform is split into
// passes over one axis at a time; every pass moves whole tiles between HBM and
// shared memory once, and the pointwise work of the method (masking by chi,
// products with u, the spectral multiply by the kernel spectrum, the final
// mask and the Verlet/damage updates) is fused into the first and last pass so
// that no field makes an extra round trip:
//
//   row pass     (x1, contiguous):  real -> packed half spectrum or back,
//                                   with a per-node prologue / epilogue;
//   column pass  (x2 or x3, strided): complex FFT over a W-column tile,
//                                   optionally forward FFT, per-mode spectral
//                                   combine of all fields, inverse FFT.
//
// Packed half spectrum: a real row of n1 samples x[0..n1) becomes n1/2
// complex values X(k), k in [0, n1/2), with slot 0 holding the two real
// values (X(0), X(n1/2)). After the column transforms, slot kx = 0 holds
// X^(0,k') + i X^(n1/2,k') for every (k2,k3); the spectral combine unpacks it
// with the mirror mode (-k2,-k3).
//
// The passes are in pd_rows.cuh and pd_cols.cuh. This file holds the Stockham
// stages of the plane passes (pd_plane.cuh: each thread owns kV = 8 complex values
// per stage, stages exchange through shared memory in autosort order, inverse
// transforms are conj DFT conj) and the compensated block sums.
#pragma once

#include <type_traits>

#include "pd_common.cuh"
#include "pd_tma.cuh"

namespace pd {

constexpr int kLgV = 3;        // log2(kV)
constexpr int kV = 1 << kLgV;  // complex values per thread and FFT stage

__host__ __device__ constexpr int bit_reverse(int i, int bits)
{
    int r = 0;
    for (int b = 0; b < bits; ++b) r |= ((i >> b) & 1) << (bits - 1 - b);
    return r;
}

// a * e^{-2 pi i m / 16}, m in [0, 8)
template <typename T>
__device__ __forceinline__ cx<T> rot16(cx<T> a, int m)
{
    const T c1 = T(0.92387953251128675613), s1 = T(0.38268343236508977173);
    const T r2 = T(0.70710678118654752440);
    switch (m) {
        case 0: return a;
        case 1: return cmul(a, mk(c1, -s1));
        case 2: return mk((a.x + a.y) * r2, (a.y - a.x) * r2);
        case 3: return cmul(a, mk(s1, -c1));
        case 4: return mk(a.y, -a.x);
        case 5: return cmul(a, mk(-s1, -c1));
        case 6: return mk((a.y - a.x) * r2, -(a.x + a.y) * r2);
        default: return cmul(a, mk(-c1, -s1));
    }
}

// Forward DFT of R values in registers (natural order in and out).
template <typename T, int R>
__device__ __forceinline__ void dft_reg(cx<T> *v)
{
    constexpr int bits = (R == 2) ? 1 : (R == 4) ? 2 : (R == 8) ? 3 : 4;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int j = bit_reverse(i, bits);
        if (i < j) {
            cx<T> t = v[i];
            v[i] = v[j];
            v[j] = t;
        }
    }
#pragma unroll
    for (int h = 1; h < R; h <<= 1) {
#pragma unroll
        for (int i = 0; i < R; i += 2 * h) {
#pragma unroll
            for (int k = 0; k < h; ++k) {
                cx<T> a = v[i + k];
                cx<T> b = rot16(v[i + k + h], k * (8 / h));
                v[i + k] = a + b;
                v[i + k + h] = a - b;
            }
        }
    }
}

// Swizzled element order between the first and second stage: element e is
// stored at e ^ ((e >> sh) & 7) (an involution for sh >= 3). The first
// radix-8 stage writes the 8 outputs of one butterfly to consecutive
// elements, so in natural order the lanes of a warp store 8 elements apart
// and pile onto two of the 16 eight-byte bank pairs; XOR-ing the element's
// low three bits with the butterfly index spreads them over all pairs. With
// 8 butterflies per row (rows 8 bank pairs apart) sh = 3 is conflict-free,
// with 16 or more sh = 4.
__device__ __forceinline__ int swz(int e, int sh) { return e ^ ((e >> sh) & 7); }

// One radix-R Stockham stage of F length-n transforms, field f stored at
// s[f * fstride + e * stride]. Thread jt (of nt = n/kV) handles butterflies
// j = jt + b nt, b < kV/R, of every field (the twiddles are loaded once for
// all fields). tw[i] = e^{-2 pi i i / 2^lgl}. SI / SO: read / write in the
// swizzled order of shift sh. Ends with a block-wide barrier.
template <typename T, int R, int F, bool SI = false, bool SO = false>
__device__ __forceinline__ void fft_stage(cx<T> *s, int fstride, int stride, int n, int ns, int lgnsr, int jt,
                                          int nt, const cx<T> *__restrict__ tw, int lgl, bool cin, bool cout,
                                          int sh = 0)
{
    static_assert(R <= kV, "radix larger than the values per thread");
    constexpr int B = kV / R;
    cx<T> v[F][kV];
    const int q = n / R;
#pragma unroll
    for (int f = 0; f < F; ++f) {
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int j = jt + b * nt;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                int e = j + r * q;
                if constexpr (SI) e = swz(e, sh);
                const cx<T> x = s[f * fstride + e * stride];
                v[f][b * R + r] = cin ? conjg(x) : x;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < B; ++b) {
        const int j = jt + b * nt;
        const int k = j & (ns - 1);
        const int o = (j - k) * R + k;
        if constexpr (F == 1) {
            if (ns > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) v[0][b * R + r] = cmul(v[0][b * R + r], tw[(r * k) << (lgl - lgnsr)]);
            }
            dft_reg<T, R>(&v[0][b * R]);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                int e = o + r * ns;
                if constexpr (SO) e = swz(e, sh);
                s[e * stride] = cout ? conjg(v[0][b * R + r]) : v[0][b * R + r];
            }
        } else {
            cx<T> w[R];
            if (ns > 1) {
#pragma unroll
                for (int r = 1; r < R; ++r) w[r] = tw[(r * k) << (lgl - lgnsr)];
            }
#pragma unroll
            for (int f = 0; f < F; ++f) {
                if (ns > 1) {
#pragma unroll
                    for (int r = 1; r < R; ++r) v[f][b * R + r] = cmul(v[f][b * R + r], w[r]);
                }
                dft_reg<T, R>(&v[f][b * R]);
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    int e = o + r * ns;
                    if constexpr (SO) e = swz(e, sh);
                    s[f * fstride + e * stride] = cout ? conjg(v[f][b * R + r]) : v[f][b * R + r];
                }
            }
        }
    }
    __syncthreads();
}

// Forward DFTs of length 2^LGN (>= 16) of F fields in shared memory, in place,
// with stage schedule SCHED (the radix-4 or radix-2 remainder stage last or
// first) and swizzle shift SH (0: none) fixed at compile time: the stage sequence unrolls, so the lengths,
// strides, twiddle shifts and conjugation flags fft_stage derives from it are
// constants (shared-memory offsets fold into the load and store instructions
// and no stage dispatch runs).
template <typename T, int F, int LGN, int SCHED, int SH, int LGNS = 0, bool SWIN = false>
__device__ __forceinline__ void fft_ct(cx<T> *s, int fstride, int stride, int jt, const cx<T> *__restrict__ tw,
                                       int lgl, bool cin, bool cout)
{
    constexpr int REM = LGN - LGNS, RM = LGN % kLgV;
    constexpr int LR = (SCHED && LGNS == 0 && RM) ? RM : (REM >= kLgV ? kLgV : REM);
    constexpr bool FIRST = LGNS == 0, LAST = REM == LR;
    constexpr bool SWOUT = kV == 8 && SH > 0 && FIRST && !LAST && LR == 3;
    fft_stage<T, (1 << LR), F, SWIN, SWOUT>(s, fstride, stride, 1 << LGN, 1 << LGNS, LGNS + LR, jt,
                                            (1 << LGN) >> kLgV, tw, lgl, cin && FIRST, cout && LAST, SH);
    if constexpr (!LAST) fft_ct<T, F, LGN, SCHED, SH, LGNS + LR, SWOUT>(s, fstride, stride, jt, tw, lgl, cin, cout);
}

// ---------------------------------------------------------------------------
// Compensated FP32 accumulation (Knuth two-sum): sums carried as an
// unevaluated pair (hi, lo), accurate to about FP32^2, so reductions run on
// FP32 units and only the block totals are combined in FP64. Inner products
// take each FP32 product exactly (the FMA residual a b - fl(a b) is itself a
// float, the error-free two-product), so a dot product of FP32 vectors is
// accumulated to about FP64 accuracy without FP64 arithmetic per element.
// ---------------------------------------------------------------------------
struct DSum {
    float hi = 0.f, lo = 0.f;
    double d = 0.0;  // FP64 operands accumulate here directly
    __device__ __forceinline__ void add(float x)
    {
        const float s = hi + x;
        const float bb = s - hi;
        lo += (hi - (s - bb)) + (x - bb);
        hi = s;
    }
    __device__ __forceinline__ void add(double x) { d += x; }
    // += a b with the product's rounding error kept
    __device__ __forceinline__ void add_prod(float a, float b)
    {
        const float p = a * b;
        lo += __fmaf_rn(a, b, -p);
        add(p);
    }
    __device__ __forceinline__ void add_prod(double a, double b) { d += a * b; }
    __device__ __forceinline__ double value() const { return d + (double)hi + (double)lo; }
};

// Sum of one double per thread over the block (all threads must call).
__device__ __forceinline__ double block_sum_d(double v)
{
    __shared__ double sh_bs[32];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh_bs[wid] = v;
    __syncthreads();
    const int nw = (blockDim.x + 31) >> 5;
    v = (threadIdx.x < nw) ? sh_bs[threadIdx.x] : 0.0;
    if (wid == 0)
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;  // valid in thread 0
}

// Block sums of NV compensated accumulators (valid in thread 0; whole warps).
// The FP32 pairs (hi, lo) are merged across each warp by the two-sum of the
// hi parts, their rounding errors going to lo, so only one lane per warp
// converts to FP64: FP64 runs at a small fraction of the FP32 rate, and a
// per-thread FP64 reduction kept that pipe busy for several microseconds of
// every row pass. FP64 parts are summed in FP64 only in warps that hold any.
template <int NV>
__device__ __forceinline__ void block_sums(const DSum *const (&a)[NV], double (&out)[NV])
{
    __shared__ double sh_bn[NV][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();  // a previous call may still be reading sh_bn
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        float hi = a[v]->hi, lo = a[v]->lo;
        double d = a[v]->d;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float h2 = __shfl_xor_sync(0xffffffffu, hi, o);
            const float l2 = __shfl_xor_sync(0xffffffffu, lo, o);
            const float s = hi + h2, bb = s - hi;
            lo += l2 + ((hi - (s - bb)) + (h2 - bb));
            hi = s;
        }
        if (__any_sync(0xffffffffu, d != 0.0))
            for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) sh_bn[v][wid] = d + (double)hi + (double)lo;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
        for (int v = 0; v < NV; ++v) {
            double t = 0.0;
            for (int k = 0; k < nw; ++k) t += sh_bn[v][k];
            out[v] = t;
        }
    }
}

}  // namespace pd

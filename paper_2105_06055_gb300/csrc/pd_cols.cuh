// Column passes of the FCBM-EC convolutions (private): transforms along x2 or
// x3 (strided axes), plain, or forward + spectral combine + inverse.
//
// What bounds them: the data moved is one read and one write of every packed
// spectrum; the arithmetic per value is small, so the cost above the traffic
// is issue slots, barriers and latency. The passes therefore hold a transform
// in registers and touch shared memory once per exchange: a length L is split
// into two (or three) radix-2^k stages, L = RA (RB) RC, decimation in
// frequency. A thread loads RA values of its column straight from global
// memory (128-byte segments across the W columns of the tile), transforms
// them in registers, writes them to shared memory, and after one barrier the
// block finishes each chunk of RC consecutive values in registers, where they
// are the modes k = q + RA (q' + RB s). The combine needs all fields of one
// mode and happens there; the inverse runs the same steps backwards on the
// same shared-memory elements (in place, mirrored order), so a forward +
// combine + inverse pass has two barriers (four with RB > 1), and no digit
// reversal is ever stored.
//
// The packed column kx = 0 (holding X(0) + i X(n1/2) of the x1 transform) is
// unpacked before the transform: with Z(k2) and its mirror Z(-k2),
//   A = (Z + conj Z(-k2)) / 2,  B = (Z - conj Z(-k2)) / (2 i)
// elementwise, since the remaining axis has not been transformed yet. The
// special tiles carry those columns as pairs (A at kx = 0, B at kx = n1/2) in
// neighbouring lanes, and write back Z = A + i B and Z(-k2) = conj A + i conj B.
// Every tile reads only what it writes, so all passes run in place.
#pragma once

#include "pd_fft.cuh"

namespace pd {

// a * e^{-+2 pi i m / 32} (forward -, inverse +), m in [0, 16)
template <typename T, bool INV>
__device__ __forceinline__ cx<T> rot32(cx<T> a, int m)
{
    constexpr double C[17] = {1.0, 0.98078528040323044913, 0.92387953251128675613, 0.83146961230254523708,
                              0.70710678118654752440, 0.55557023301960222474, 0.38268343236508977173,
                              0.19509032201612826785, 0.0, -0.19509032201612826785, -0.38268343236508977173,
                              -0.55557023301960222474, -0.70710678118654752440, -0.83146961230254523708,
                              -0.92387953251128675613, -0.98078528040323044913, -1.0};
    if (m == 0) return a;
    if (m == 8) return INV ? mk(-a.y, a.x) : mk(a.y, -a.x);
    const T c = (T)C[m], s = (T)(m <= 8 ? C[8 - m] : C[m - 8]);  // sin = cos(pi/2 - .)
    if (m == 4) return INV ? mk((a.x - a.y) * c, (a.x + a.y) * c) : mk((a.x + a.y) * c, (a.y - a.x) * c);
    if (m == 12) return INV ? mk((a.x + a.y) * c, (a.y - a.x) * c) : mk((a.y - a.x) * -c, (a.x + a.y) * c);
    return INV ? mk(a.x * c - a.y * s, a.y * c + a.x * s) : mk(a.x * c + a.y * s, a.y * c - a.x * s);
}

// DFT of R values in registers, natural order in and out (e^{-...} or, INV, e^{+...}).
template <typename T, int R, bool INV>
__device__ __forceinline__ void dft_n(cx<T> *v)
{
    constexpr int bits = R == 1 ? 0 : R == 2 ? 1 : R == 4 ? 2 : R == 8 ? 3 : R == 16 ? 4 : 5;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int j = bit_reverse(i, bits);
        if (i < j) {
            const cx<T> t = v[i];
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
                const cx<T> a = v[i + k];
                const cx<T> b = rot32<T, INV>(v[i + k + h], k * (16 / h));
                v[i + k] = a + b;
                v[i + k + h] = a - b;
            }
        }
    }
}

// Shape of a pass of length 2^LG over FB fields: chunk radix 2^LGC, largest
// first-stage radix 2^LGM.
template <typename T, int LG, int FB, int LGC_, int LGM, int WMIN = 64, int WMAX = 128>
struct ColShape {
    static constexpr int LGC = LGC_ < LG ? LGC_ : LG;
    static constexpr int REM = LG - LGC;
    static constexpr int LGA = REM <= LGM ? REM : (REM - LGM <= LGM ? LGM : (REM + 1) / 2);
    static constexpr int LGB = REM - LGA;
    static constexpr int LGV = LGA > LGB ? (LGA > LGC ? LGA : LGC) : (LGB > LGC ? LGB : LGC);
    static constexpr int L = 1 << LG, RA = 1 << LGA, RB = 1 << LGB, RC = 1 << LGC, V = 1 << LGV;
    static constexpr int NT = L / V;  // threads per column and field group
    static constexpr int M = L / RA;  // first-stage stride
    // Field groups: with many fields the stages run on separate fields in
    // parallel (each group takes every G-th field) and the chunks are shared out
    static constexpr int G = FB >= 12 && V / RC >= 8 ? 8 : FB >= 5 && V / RC >= 4 ? 4 : FB >= 5 && V / RC >= 2 ? 2 : 1;
    static constexpr int LGP = LGC < 3 ? 3 : LGC;  // rows per pad row
    static constexpr size_t col_bytes(int pad) { return (size_t)FB * (L + (pad ? L >> LGP : 0)) * sizeof(cx<T>); }
    // Tile width: 128-byte segments while three blocks of the tile fit on an SM
    // (whole warps at least), then narrower, down to WMIN bytes: 64 for 3D boxes
    // (512^3, 32-byte segments: 2840 us a pass, 64-byte: 1544). WMAX and WMIN are
    // 32 for the cache-resident 2D grids, where more tiles fill more SMs
    static constexpr int width()
    {
        int w = (int)(WMAX / sizeof(cx<T>));
        while (w * NT * G < 32) w <<= 1;
        while (w * (int)sizeof(cx<T>) > WMIN && (col_bytes(0) * w > 70 * 1024 || w * NT * G > 512)) w >>= 1;
        while (w > 2 && col_bytes(1) * w > 220 * 1024) w >>= 1;
        return w;
    }
    static constexpr int W = width();
    static constexpr int LGW = W == 16 ? 4 : W == 8 ? 3 : W == 4 ? 2 : 1;
    // rows narrower than the 32 banks: one pad row per chunk keeps the chunk
    // accesses of neighbouring lanes on different banks (chunks of 4: one per two
    // chunks, so that two blocks of the 12-field pass fit on an SM)
    static constexpr bool PAD = W * sizeof(cx<T>) < 128 && RC >= 4;
    static constexpr int THREADS = W * NT * G;
    static constexpr int FSZ = (L + (PAD ? L >> LGP : 0)) * W;  // field stride in shared memory
    static constexpr size_t smem = (size_t)FB * FSZ * sizeof(cx<T>);
    static_assert(W * NT * G >= 32, "whole warps");
    __device__ static __forceinline__ int at(int loc, int c) { return ((PAD ? loc + (loc >> LGP) : loc) << LGW) + c; }
};

template <typename T>
struct ColArgs {
    cx<T> *spec;
    int64_t fs;   // slot stride
    int64_t ls;   // stride along the transformed axis
    int64_t os;   // stride of the outer axis (blockIdx.y)
    int lgh;      // log2(n1/2)
    int n2;       // 3D last axis: n2; 2D last axis: 1 (one kx = 0 column, its own mirror)
    int nspec;    // special tiles (first blocks; 0 for the plain passes)
    int sw;       // columns of a special tile on long axes (special_cols)
    int zaxis;    // 1: the transformed axis is x3
};

// Twiddle tables of a plan, for every length 2^lg up to the longest axis: the
// plain table W^i (lga = 0), and for the stages of radix 2^lga the table
// W^{j q} at j 2^lga + q, so that a butterfly's twiddles are consecutive
// (16-byte loads, no index arithmetic per value).
constexpr int kTwRadices = 6;  // lga = 0 ... 5
__host__ __device__ constexpr int tw_base(int lg, int lga) { return kTwRadices * ((1 << lg) - 1) + (lga << lg); }
__host__ __device__ constexpr int tw_entries(int lgmax) { return tw_base(lgmax + 1, 0); }

template <typename T>
__device__ __forceinline__ cx<T> ldg_cx(const cx<T> *p)
{
    if constexpr (sizeof(T) == 4) {
        const float2 v = __ldg(reinterpret_cast<const float2 *>(p));
        return mk((T)v.x, (T)v.y);
    } else {
        const double2 v = __ldg(reinterpret_cast<const double2 *>(p));
        return mk((T)v.x, (T)v.y);
    }
}
// W_{2^LG}^i
template <typename T, int LG>
__device__ __forceinline__ cx<T> twid(const cx<T> *__restrict__ tw, unsigned i)
{
    return ldg_cx(tw + tw_base(LG, 0) + i);
}
// v[q] *= W_{2^LG}^{j q} (or its conjugate), q = 1 ... 2^LGR - 1
template <typename T, int LG, int LGR, bool CONJ>
__device__ __forceinline__ void twiddle(cx<T> *v, int j, const cx<T> *__restrict__ tw)
{
    constexpr int R = 1 << LGR;
    const cx<T> *p = tw + tw_base(LG, LGR) + ((unsigned)j << LGR);
#pragma unroll
    for (int q = 0; q < R; q += 2) {
        cx<T> w0, w1;
        if constexpr (sizeof(T) == 4) {
            const float4 w = __ldg(reinterpret_cast<const float4 *>(p + q));
            w0 = mk((T)w.x, (T)w.y);
            w1 = mk((T)w.z, (T)w.w);
        } else {
            w0 = q ? ldg_cx(p + q) : mk(T(1), T(0));
            w1 = ldg_cx(p + q + 1);
        }
        if (q) v[q] = cmul(v[q], CONJ ? conjg(w0) : w0);
        v[q + 1] = cmul(v[q + 1], CONJ ? conjg(w1) : w1);
    }
}

// one first-stage butterfly after its loads: DFT over r, twiddle W_L^{j q}
template <typename T, class S, int LG>
__device__ __forceinline__ void stage_a(cx<T> *v, int j, const cx<T> *__restrict__ tw)
{
    dft_n<T, S::RA, false>(v);
    if constexpr (S::M > 1 && S::LGA > 0) twiddle<T, LG, S::LGA, false>(v, j, tw);
}
// its inverse: conjugate twiddle, inverse DFT over q
template <typename T, class S, int LG>
__device__ __forceinline__ void stage_a_inv(cx<T> *v, int j, const cx<T> *__restrict__ tw)
{
    if constexpr (S::M > 1 && S::LGA > 0) twiddle<T, LG, S::LGA, true>(v, j, tw);
    dft_n<T, S::RA, true>(v);
}
// middle stage of one field, in place in shared memory
template <typename T, class S, int LG, bool INV>
__device__ __forceinline__ void stage_b(cx<T> *s, int c, int jt, const cx<T> *__restrict__ tw)
{
#pragma unroll
    for (int b = 0; b < S::V / S::RB; ++b) {
        const int i = jt + b * S::NT, j = i & (S::RC - 1), q = i >> S::LGC;
        cx<T> v[S::RB];
#pragma unroll
        for (int r = 0; r < S::RB; ++r) v[r] = s[S::at(q * S::M + r * S::RC + j, c)];
        if constexpr (INV) twiddle<T, LG - S::LGA, S::LGB, true>(v, j, tw);
        dft_n<T, S::RB, INV>(v);
        if constexpr (!INV) twiddle<T, LG - S::LGA, S::LGB, false>(v, j, tw);
#pragma unroll
        for (int r = 0; r < S::RB; ++r) s[S::at(q * S::M + r * S::RC + j, c)] = v[r];
    }
}
// mode of value s of chunk ch = q RB + q'
template <class S>
__device__ __forceinline__ int chunk_mode(int ch, int s)
{
    const int q = ch >> S::LGB, q2 = ch & (S::RB - 1);
    return q + (q2 << S::LGA) + (s << (S::LGA + S::LGB));
}

// Plain transform along x2 of one field per block: grid (tiles, outer, fields).
template <typename T, int LG, bool INV>
struct PlainShape : ColShape<T, LG, 1, (LG >= 8 ? 4 : 3), (sizeof(T) == 4 ? 5 : 4)> {
};
template <typename T, int LG, bool INV>
__global__ void __launch_bounds__(PlainShape<T, LG, INV>::THREADS)
    k_col_plain(ColArgs<T> g, int slot0, const cx<T> *__restrict__ tw)
{
    using S = PlainShape<T, LG, INV>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<T> *s = reinterpret_cast<cx<T> *>(smem_raw);
    const int c = threadIdx.x & (S::W - 1), jt = threadIdx.x >> S::LGW;
    // uniform base + 32-bit lane offset (a slot is below 2^32 values)
    cx<T> *p = g.spec + (slot0 + (int)blockIdx.z) * g.fs + blockIdx.y * g.os + (int64_t)blockIdx.x * S::W;
    const unsigned ls = (unsigned)g.ls;
    pdl_wait();
    auto chunk_pass = [&]() {
#pragma unroll
        for (int b = 0; b < S::V / S::RC; ++b) {
            const int ch = jt + b * S::NT;
            const unsigned off = (unsigned)chunk_mode<S>(ch, 0) * ls + c;
            constexpr unsigned K = S::L / S::RC;  // mode step within a chunk
            cx<T> v[S::RC];
#pragma unroll
            for (int k = 0; k < S::RC; ++k) v[k] = INV ? (p + k * K * ls)[off] : s[S::at(ch * S::RC + k, c)];
            dft_n<T, S::RC, INV>(v);
#pragma unroll
            for (int k = 0; k < S::RC; ++k) {
                if constexpr (INV)
                    s[S::at(ch * S::RC + k, c)] = v[k];
                else
                    (p + k * K * ls)[off] = v[k];
            }
        }
    };
    auto first_pass = [&]() {
#pragma unroll
        for (int b = 0; b < S::V / S::RA; ++b) {
            const int j = jt + b * S::NT;
            const unsigned off = j * ls + c;
            cx<T> v[S::RA];
#pragma unroll
            for (int r = 0; r < S::RA; ++r) v[r] = INV ? s[S::at(j + r * S::M, c)] : (p + r * S::M * ls)[off];
            if constexpr (INV)
                stage_a_inv<T, S, LG>(v, j, tw);
            else
                stage_a<T, S, LG>(v, j, tw);
#pragma unroll
            for (int r = 0; r < S::RA; ++r) {
                if constexpr (INV)
                    (p + r * S::M * ls)[off] = v[r];
                else
                    s[S::at(j + r * S::M, c)] = v[r];
            }
        }
    };
    if constexpr (INV)
        chunk_pass();
    else
        first_pass();
    __syncthreads();
    if constexpr (S::RB > 1) {
        stage_b<T, S, LG, INV>(s, c, jt, tw);
        __syncthreads();
    }
    if constexpr (INV)
        first_pass();
    else
        chunk_pass();
}

// Chunk radix of a combining pass: the chunk's values of all fields live in
// registers between the two chunk transforms (2 FB RC words)
template <typename T, int FB>
constexpr int comb_lgc()
{
    const int words = FB * (sizeof(T) == 4 ? 2 : 4);
    return words * 8 <= 96 ? 3 : words * 4 <= 96 ? 2 : words * 2 <= 96 ? 1 : 0;
}
template <typename T, class Op, int LG>
struct CombShape
    : ColShape<T, LG, (Op::kFin > Op::kFout ? Op::kFin : Op::kFout),
               comb_lgc<T, (Op::kFin > Op::kFout ? Op::kFin : Op::kFout)>(), 3, Op::kDim == 2 ? 32 : 64, Op::kDim == 2 ? 32 : 128> {
};
// Resident blocks the register allocation has to allow: 128 registers (FP64:
// 168) or what shared memory allows. Measured at 256^3: radix-8 first stages
// at 128 registers 153 us, radix 16 at 168 registers 168 us (fewer warps) and at
// 128 registers 216 us, radix 8 capped at 80 registers 172 us and at 64 250 us.
template <typename T, class S>
constexpr int comb_blocks()
{
    int n = 65536 / (S::THREADS * (sizeof(T) == 4 ? 128 : 168));
    const int m = (int)(227 * 1024 / (S::smem + 1024));
    n = n < m ? n : m;
    return n < 1 ? 1 : n;
}

// Columns of a special tile (pairs): their elements are scattered 8- or 16-byte words
// (one L1 lookup each), so they are spread over more blocks than whole tiles
// would make; with 16 columns these few blocks ran three times as long as the
// others and set the pass's time at 128^3. On long axes of boxes whose other tiles fit
// the SMs at once they still did with four (force on 32 x 16 x 1024 nodes in FP32: 84
// us, with one pair a block 65, before the passes were rewritten 63; 32 x 16 x 512: 41.5
// and 33.5): those take one pair. With more tiles the special ones end under the
// others, and twice as many cost time (64 x 128 x 1024: 353 us, with one pair 368).
// Below 512 nodes the two forms differ by a few us.
constexpr int kSpecCols = 4, kLgLong = 9;
__host__ __device__ constexpr int special_cols(int lg, int width, int64_t tiles, int nsm)
{
    return lg >= kLgLong && tiles <= nsm ? 2 : width < kSpecCols ? width : kSpecCols;
}

// Op of a combining pass:
//   static constexpr int kFin, kFout, kTab;
//   int slot_in(int f), slot_out(int f): packed-spectrum slots
//   const T *table(int c): kTab folded kernel-spectrum components
//        ([k3f][k2f][k1], k1 in [0, n1/2])
//   void combine(const T *t, bool fy, bool fz, const cx<T> *in, cx<T> *out):
//        t: the mode's kTab table values; fy / fz: k2 / k3 were folded to n - k
template <typename T, class Op, int LG>
__global__ void __launch_bounds__(CombShape<T, Op, LG>::THREADS, comb_blocks<T, CombShape<T, Op, LG>>())
    k_col_comb(ColArgs<T> g, Op op, const cx<T> *__restrict__ tw)
{
    using S = CombShape<T, Op, LG>;
    constexpr int FI = Op::kFin, FO = Op::kFout, FB = FI > FO ? FI : FO;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<T> *sm = reinterpret_cast<cx<T> *>(smem_raw);
    const int c = threadIdx.x & (S::W - 1);
    const int jg = threadIdx.x >> S::LGW;                                  // chunk owner, [0, NT G)
    const int jt = S::G > 1 ? jg % S::NT : jg, fg = S::G > 1 ? jg / S::NT : 0;  // column thread, field group
    const int H = 1 << g.lgh;
    const bool special = (int)blockIdx.x < g.nspec;
    // this lane's column: element offset (and its mirror's), kx and ky
    unsigned col, mir = 0;  // (a slot is below 2^32 values)
    int kx, ky;
    bool active;
    if (special) {
        const int sw = Op::kDim == 3 && LG >= kLgLong ? g.sw : special_cols(0, S::W, 0, 0);
        const int cc = (int)blockIdx.x * sw + c, k2 = cc >> 1;
        active = c < sw && k2 <= (g.n2 >> 1);
        ky = active ? k2 : 0;
        kx = (cc & 1) ? H : 0;
        col = (unsigned)ky << g.lgh;
        mir = (unsigned)((g.n2 - ky) & (g.n2 - 1)) << g.lgh;
    } else {
        col = (unsigned)((int)blockIdx.x - g.nspec) * S::W + c;
        kx = (int)(col & (H - 1));
        ky = (int)(col >> g.lgh);
        active = kx != 0;
    }
    const unsigned ls = (unsigned)g.ls;
    const int64_t step = (int64_t)S::M * ls;
    pdl_wait();

    // first stage: global -> registers -> shared. With few fields all of a
    // thread's loads are issued before the first value is used.
    constexpr int NV = S::V / S::RA;
    auto load = [&](cx<T> *v, int f, int j) {
        const cx<T> *p = g.spec + op.slot_in(f) * g.fs;
        if (special) {
#pragma unroll
            for (int r = 0; r < S::RA; ++r) {
                cx<T> z = mk(T(0), T(0)), y = z;
                if (active) {
                    z = (p + r * step)[col + j * ls];
                    y = (p + r * step)[mir + j * ls];
                }
                v[r] = kx ? mk(T(0.5) * (z.y + y.y), T(0.5) * (y.x - z.x))
                          : mk(T(0.5) * (z.x + y.x), T(0.5) * (z.y - y.y));
            }
        } else {
#pragma unroll
            for (int r = 0; r < S::RA; ++r) v[r] = active ? (p + r * step)[col + j * ls] : mk(T(0), T(0));
        }
    };
    auto first = [&](cx<T> *v, int f, int j) {
        stage_a<T, S, LG>(v, j, tw);
#pragma unroll
        for (int r = 0; r < S::RA; ++r) sm[f * S::FSZ + S::at(j + r * S::M, c)] = v[r];
    };
    if constexpr (S::G == 1 && FI * S::V * sizeof(T) <= 3 * 16 * 4) {
        cx<T> v[FI][NV][S::RA];
#pragma unroll
        for (int f = 0; f < FI; ++f)
#pragma unroll
            for (int b = 0; b < NV; ++b) load(v[f][b], f, jt + b * S::NT);
#pragma unroll
        for (int f = 0; f < FI; ++f)
#pragma unroll
            for (int b = 0; b < NV; ++b) first(v[f][b], f, jt + b * S::NT);
    } else {
#pragma unroll 1
        for (int f = fg; f < FI; f += S::G) {
            cx<T> v[NV][S::RA];
#pragma unroll
            for (int b = 0; b < NV; ++b) load(v[b], f, jt + b * S::NT);
#pragma unroll
            for (int b = 0; b < NV; ++b) first(v[b], f, jt + b * S::NT);
        }
    }
    __syncthreads();
    if constexpr (S::RB > 1) {
#pragma unroll 1
        for (int f = fg; f < FI; f += S::G) stage_b<T, S, LG, false>(sm + f * S::FSZ, c, jt, tw);
        __syncthreads();
    }

    // chunks: finish the forward transform, combine the fields mode by mode,
    // start the inverse; in place
    {
        constexpr int half = S::L / 2;
        const int kyf = ky > (g.n2 >> 1) ? g.n2 - ky : ky;
        const unsigned rs = (unsigned)(H + 1) * (g.zaxis ? (unsigned)((g.n2 >> 1) + 1) : 1u);
        const unsigned tcol = (g.zaxis ? (unsigned)kyf * (H + 1) : 0u) + kx;
#pragma unroll 1
        for (int b = 0; b < S::V / S::RC / S::G; ++b) {
            const int ch = jg + b * S::NT * S::G;
            T t[S::RC][Op::kTab];
#pragma unroll
            for (int k = 0; k < S::RC; ++k) {
                const int mode = chunk_mode<S>(ch, k);
                const unsigned ti = (unsigned)(mode > half ? S::L - mode : mode) * rs + tcol;
#pragma unroll
                for (int q = 0; q < Op::kTab; ++q) t[k][q] = __ldg(op.table(q) + ti);
            }
            cx<T> v[FB][S::RC];
#pragma unroll
            for (int f = 0; f < FI; ++f) {
#pragma unroll
                for (int k = 0; k < S::RC; ++k) v[f][k] = sm[f * S::FSZ + S::at(ch * S::RC + k, c)];
                dft_n<T, S::RC, false>(v[f]);
            }
#pragma unroll
            for (int k = 0; k < S::RC; ++k) {
                const bool fr = chunk_mode<S>(ch, k) > half;
                cx<T> in[FI], out[FO];
#pragma unroll
                for (int f = 0; f < FI; ++f) in[f] = v[f][k];
                op.combine(t[k], g.zaxis ? ky > (g.n2 >> 1) : fr, g.zaxis && fr, in, out);
#pragma unroll
                for (int f = 0; f < FO; ++f) v[f][k] = out[f];
            }
#pragma unroll
            for (int f = 0; f < FO; ++f) {
                dft_n<T, S::RC, true>(v[f]);
#pragma unroll
                for (int k = 0; k < S::RC; ++k) sm[f * S::FSZ + S::at(ch * S::RC + k, c)] = v[f][k];
            }
        }
    }
    __syncthreads();
    if constexpr (S::RB > 1) {
#pragma unroll 1
        for (int f = fg; f < FO; f += S::G) stage_b<T, S, LG, true>(sm + f * S::FSZ, c, jt, tw);
        __syncthreads();
    }

    // last stage: shared -> registers -> global
#pragma unroll 1
    for (int f = fg; f < FO; f += S::G) {
        cx<T> *p = g.spec + op.slot_out(f) * g.fs;
        const cx<T> *s = sm + f * S::FSZ;
#pragma unroll
        for (int b = 0; b < S::V / S::RA; ++b) {
            const int j = jt + b * S::NT;
            cx<T> v[S::RA];
#pragma unroll
            for (int r = 0; r < S::RA; ++r) v[r] = s[S::at(j + r * S::M, c)];
            stage_a_inv<T, S, LG>(v, j, tw);
            if (special) {
                // lane pairs hold A and B: the even lane writes A + i B, the
                // odd one the mirror column conj A + i conj B
                const bool wr = active && !(kx && mir == col);
                const unsigned d = (kx ? mir : col) + j * ls;
                const unsigned two = 3u << (threadIdx.x & 30);  // the lane pair
#pragma unroll
                for (int r = 0; r < S::RA; ++r) {
                    const cx<T> o = mk(__shfl_xor_sync(two, v[r].x, 1), __shfl_xor_sync(two, v[r].y, 1));
                    const cx<T> z = kx ? mk(o.x + v[r].y, v[r].x - o.y) : mk(v[r].x - o.y, v[r].y + o.x);
                    if (wr) (p + r * step)[d] = z;
                }
            } else if (active) {
#pragma unroll
                for (int r = 0; r < S::RA; ++r) (p + r * step)[col + j * ls] = v[r];
            }
        }
    }
}

}  // namespace pd

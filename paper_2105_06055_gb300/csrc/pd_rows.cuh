// Row passes of the FCBM-EC convolutions (private): real transforms along x1
// (contiguous rows) with the per-node work of the method fused in front of the
// forward transform or behind the inverse one.
//
// What bounds them: the node fields and the packed spectra are moved once; the
// rest is latency (dependent loads of the node work, exchanges between the
// transform's stages), so the passes are cut into many small independent
// pieces. A block takes a few rows (as many as one warp transforms at a time)
// of all fields. The transforms are warp-wide: NT lanes (H/16 or H/8) hold a row of
// H packed values, the lanes of a warp 32/NT rows of one field, and a warp's
// stages exchange through its own rows of shared memory with warp barriers
// only. One block barrier separates the node work (all lanes over consecutive
// nodes, all fields of a node in one lane) from the transforms (one field per
// warp). A lane finishes the chunks of modes m + s K and (K - m) + s K (K
// chunks), which hold each other's mirror modes, so the real-transform unpack
// happens in registers.
//
// Spectra move between global and shared memory by bulk copies, one per row:
// the lanes' own accesses (8 rows, four to eight modes each, and the mirrored
// ones) made 8 to 16 L1 lookups per instruction, and L1 lookups set the pace of
// the passes (88% busy at 256^3).
//
// Between the stages a row carries one pad element per chunk, and the row pitch
// puts the rows of a warp on different banks, which makes the strided stage
// accesses and the chunk accesses conflict-free. Spectra lie in natural order at
// the front of the same row.
#pragma once

#include <type_traits>

#include "pd_cols.cuh"

namespace pd {

// Chunk radix (log2) of a row of 2^lg packed values: 8, a lane then holds 16
// values; 4 (8 values a lane, twice the lanes per row) for FP64 and for the 2D
// grids up to 512 nodes wide. Both have few warps for the chip otherwise: a
// 128 x 128 plate in FP64 has 256 row transforms, and a warp's FP64 instructions
// ran one after the other on 8 of the SMs (force 71 us, now 53; 512 x 128: 102,
// now 79; 512 x 1024 in FP32: 43, now 35).
__host__ __device__ constexpr int row_lgc(bool fp64, int dim, int lg) { return (fp64 || dim == 2) && lg <= 8 ? 2 : 3; }

// Lanes of a row: one row of 1024 packed values takes two warps (a named barrier
// in place of the warp barrier), all others a warp or part of one. With 32 values
// per lane the passes were a chain of one warp's instructions (force 2048 x 64 28 us,
// now 20; 2048 x 512 43, now 36).
__host__ __device__ constexpr int row_lanes(int H, int lgc)
{
    return (H >> (lgc + 1)) < 32 ? H >> (lgc + 1) : H >= 1024 ? 64 : 32;
}
// barrier of the lanes of a row (and of the other rows of their warp)
template <int NT>
__device__ __forceinline__ void row_sync()
{
    if constexpr (NT > 32)
        asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / NT), "n"(NT) : "memory");
    else
        __syncwarp();
}

// Row transform of 2^LG packed values: stages RA (RB) RC.
template <int LG, int LGC_>
struct RowShape {
    static constexpr int H = 1 << LG;
    static constexpr int LGC = LGC_, RC = 1 << LGC;
    static constexpr int NT = row_lanes(H, LGC);  // lanes per row
    static constexpr int V = H / NT;
    static constexpr int REM = LG - LGC, LGV = LG - (NT == 64 ? 6 : NT == 32 ? 5 : LG - LGC - 1);
    static constexpr int LGA = REM <= LGV && REM <= 4 ? REM : (REM + 1) / 2;
    static constexpr int LGB = REM - LGA;
    static constexpr int RA = 1 << LGA, RB = 1 << LGB, M = H / RA, K = H / RC;
    static constexpr int MP = M + M / RC;  // first-stage stride with the pad elements
    static constexpr int PAIRS = K / 2 / NT;
    static_assert(LG >= 4 && LG <= 10 && PAIRS >= 1 && RA <= V && RB <= V && M % RC == 0, "row length");
};
// pitch of a padded row in shared memory (complex elements; even: rows start on
// 16-byte boundaries), rows of a warp or of a pair of warps
__host__ __device__ constexpr int row_pitch(int H, int lgc)
{
    const int nt = row_lanes(H, lgc);
    return H + (H >> lgc) + (nt >= 16 ? 0 : nt == 1 ? 2 : nt);
}
__host__ __device__ constexpr int row_warp_rows(int H, int lgc) { return row_lanes(H, lgc) < 32 ? 32 / row_lanes(H, lgc) : 1; }
template <int LGC>
__device__ __forceinline__ int row_at(int e)
{
    return e + (e >> LGC);
}
// a tile holds the rows one warp transforms at a time, more of them for one
// or two fields, and a warp (or pair) per field and such group, up to twelve warps.
// Two fields in FP64 and rows of 1024 packed values take one group: a block's warps
// share one FP64 pipe and a grid of few rows has few blocks (2048 x 16: FP64 132 us
// with two groups, 85 with one, 99 before the passes were rewritten; FP32 22.0, 18.3,
// 17.9; larger grids at least as fast). FP32 rows of up to 512 keep two (1024 x 512
// fracture steps: 1234 us, with one 1271).
__host__ __device__ constexpr int row_groups(bool fp64, int H, int lgc, int fields)
{
    return fields == 1 ? 4 : fields == 2 && lgc == 3 && !fp64 && H < 1024 ? 2 : 1;
}
__host__ __device__ constexpr int row_tile_rows(bool fp64, int H, int lgc, int fields)
{
    return row_warp_rows(H, lgc) * row_groups(fp64, H, lgc, fields);
}
__host__ __device__ constexpr int row_warps(bool fp64, int H, int lgc, int fields)
{
    const int tasks = fields * row_groups(fp64, H, lgc, fields), pair = row_lanes(H, lgc) > 32 ? 2 : 1;
    int w = tasks;
    for (int k = 2; w * pair > 12; ++k) w = (tasks + k - 1) / k;
    return w * pair;
}

// chunk index (shared-memory order) of mode residue m: m = q + RA q', chunk q RB + q'
template <class S>
__device__ __forceinline__ int row_chunk(int m)
{
    return ((m & (S::RA - 1)) << S::LGB) + (m >> S::LGA);
}

// middle stage of a row (H >= 256), in place
template <typename T, class S, int LG, bool INV>
__device__ __forceinline__ void row_stage_b(cx<T> *s, int t, const cx<T> *__restrict__ tw)
{
#pragma unroll
    for (int b = 0; b < S::V / S::RB; ++b) {
        const int i = t + b * S::NT, j = i & (S::RC - 1), o = (i >> S::LGC) * S::MP + j;
        cx<T> v[S::RB];
#pragma unroll
        for (int r = 0; r < S::RB; ++r) v[r] = s[o + r * (S::RC + 1)];
        if constexpr (INV) twiddle<T, LG - S::LGA, S::LGB, true>(v, j, tw);
        dft_n<T, S::RB, INV>(v);
        if constexpr (!INV) twiddle<T, LG - S::LGA, S::LGB, false>(v, j, tw);
#pragma unroll
        for (int r = 0; r < S::RB; ++r) s[o + r * (S::RC + 1)] = v[r];
    }
}

// Forward transform of one packed row in shared memory (so: this lane's row) to
// the packed half spectrum, in place; all lanes of the warp call, those without
// a row (grids with fewer rows than a warp holds) with on = false.
template <typename T, int LG, int LGC>
__device__ __forceinline__ void row_forward(unsigned so, bool on, int t, const cx<T> *__restrict__ tw)
{
    using S = RowShape<LG, LGC>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<T> *s = reinterpret_cast<cx<T> *>(smem_raw + so);
#pragma unroll
    for (int b = 0; on && b < S::V / S::RA; ++b) {
        const int j = t + b * S::NT, o = row_at<LGC>(j);
        cx<T> v[S::RA];
#pragma unroll
        for (int r = 0; r < S::RA; ++r) v[r] = s[o + r * S::MP];
        dft_n<T, S::RA, false>(v);
        twiddle<T, LG, S::LGA, false>(v, j, tw);
#pragma unroll
        for (int r = 0; r < S::RA; ++r) s[o + r * S::MP] = v[r];
    }
    row_sync<S::NT>();
    if constexpr (S::RB > 1) {
        if (on) row_stage_b<T, S, LG, false>(s, t, tw);
        row_sync<S::NT>();
    }
    // all chunks into registers before the spectrum overwrites them
    cx<T> z[S::PAIRS][S::RC], y[S::PAIRS][S::RC];
#pragma unroll
    for (int b = 0; on && b < S::PAIRS; ++b) {
        const int m = t + b * S::NT;             // 0 <= m < K/2
        const int mm = m ? S::K - m : S::K / 2;  // its partner (m = 0: the other self-mirrored residue)
        const int ca = row_chunk<S>(m) * (S::RC + 1), cb = row_chunk<S>(mm) * (S::RC + 1);
#pragma unroll
        for (int k = 0; k < S::RC; ++k) z[b][k] = s[ca + k];
#pragma unroll
        for (int k = 0; k < S::RC; ++k) y[b][k] = s[cb + k];
    }
    row_sync<S::NT>();
#pragma unroll
    for (int b = 0; on && b < S::PAIRS; ++b) {
        const int m = t + b * S::NT;
        dft_n<T, S::RC, false>(z[b]);
        dft_n<T, S::RC, false>(y[b]);
        // Mode pairs (k, H - k): for m > 0 (z[k], y[RC-1-k]) at m + K k; the lane
        // of m = 0 holds both self-mirrored residues and pairs (y[k], y[RC-1-k])
        // at K/2 + K k for k < RC/2 and (z[k], z[RC-k]) at K k above.
        // With s = Z(k) + conj Z(H-k), t = W^k (Z(k) - conj Z(H-k)):
        //   X(k) = (s - i t) / 2,  X(H-k) = conj(s + i t) / 2
        constexpr int C2 = S::RC / 2;
        const int lo = m ? m : S::K / 2;
        const T half = T(0.5);
        if (!m) s[0] = mk(z[b][0].x + z[b][0].y, z[b][0].x - z[b][0].y);
#pragma unroll
        for (int k = 0; k < S::RC; ++k) {
            cx<T> a = z[b][k], c = y[b][S::RC - 1 - k];
            if (k < C2) {
                a.x = m ? a.x : y[b][k].x;
                a.y = m ? a.y : y[b][k].y;
            } else {
                c.x = m ? c.x : z[b][S::RC - k].x;
                c.y = m ? c.y : z[b][S::RC - k].y;
            }
            const int mode = (k < C2 ? lo : m) + S::K * k;
            const cx<T> w = scale(twid<T, LG + 1>(tw, mode), half);
            const T sx = half * (a.x + c.x), sy = half * (a.y - c.y);
            const cx<T> u = cmul(w, mk(a.x - c.x, a.y + c.y));
            s[mode] = mk(sx + u.y, sy - u.x);
            s[S::H - mode] = mk(sx - u.y, -(sy + u.x));
        }
    }
}

// Inverse transform of a packed half spectrum in shared memory to the packed
// row, in place: x[2n] = Re, x[2n+1] = Im (unnormalised).
template <typename T, int LG, int LGC>
__device__ __forceinline__ void row_inverse(unsigned so, bool on, int t, const cx<T> *__restrict__ tw)
{
    using S = RowShape<LG, LGC>;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    cx<T> *s = reinterpret_cast<cx<T> *>(smem_raw + so);
    constexpr int C2 = S::RC / 2;
    cx<T> a[S::PAIRS][S::RC], c[S::PAIRS][S::RC], x0 = mk(T(0), T(0));
#pragma unroll
    for (int b = 0; on && b < S::PAIRS; ++b) {
        const int m = t + b * S::NT, lo = m ? m : S::K / 2;
        if (b == 0 && !m) x0 = s[0];
#pragma unroll
        for (int k = 0; k < S::RC; ++k) a[b][k] = s[(k < C2 ? lo : m) + S::K * k];
#pragma unroll
        for (int k = 0; k < S::RC; ++k) c[b][k] = s[S::H - ((k < C2 ? lo : m) + S::K * k)];
    }
    row_sync<S::NT>();  // the spectrum is in registers; the chunks overwrite it
#pragma unroll
    for (int b = 0; on && b < S::PAIRS; ++b) {
        const int m = t + b * S::NT, lo = m ? m : S::K / 2, mm = m ? S::K - m : S::K / 2;
        const int ca = row_chunk<S>(m) * (S::RC + 1), cb = row_chunk<S>(mm) * (S::RC + 1);
        // the mode pairs of row_forward; with s = X(k) + conj X(H-k),
        // t = conj(W^k) (X(k) - conj X(H-k)):  Z(k) = s + i t, Z(H-k) = conj(s - i t)
#pragma unroll
        for (int k = 0; k < S::RC; ++k) {
            const cx<T> w = conjg(twid<T, LG + 1>(tw, (k < C2 ? lo : m) + S::K * k));
            const cx<T> p = a[b][k], q = c[b][k];
            const T sx = p.x + q.x, sy = p.y - q.y;
            const cx<T> u = cmul(w, mk(p.x - q.x, p.y + q.y));
            a[b][k] = mk(sx - u.y, sy + u.x);
            c[b][k] = mk(sx + u.y, u.x - sy);
        }
        cx<T> z[S::RC], y[S::RC];
        const cx<T> z0 = mk(x0.x + x0.y, x0.x - x0.y);
#pragma unroll
        for (int k = 0; k < S::RC; ++k) {
            if (k < C2) {
                const cx<T> p = k ? c[b][S::RC - k] : z0, q = c[b][S::RC - 1 - k];
                z[k] = mk(m ? a[b][k].x : p.x, m ? a[b][k].y : p.y);
                y[k] = mk(m ? q.x : a[b][k].x, m ? q.y : a[b][k].y);
            } else {
                z[k] = a[b][k];
                y[k] = c[b][S::RC - 1 - k];
            }
        }
        dft_n<T, S::RC, true>(z);
        dft_n<T, S::RC, true>(y);
#pragma unroll
        for (int k = 0; k < S::RC; ++k) s[ca + k] = z[k];
#pragma unroll
        for (int k = 0; k < S::RC; ++k) s[cb + k] = y[k];
    }
    row_sync<S::NT>();
    if constexpr (S::RB > 1) {
        if (on) row_stage_b<T, S, LG, true>(s, t, tw);
        row_sync<S::NT>();
    }
    if (!on) return;
#pragma unroll
    for (int b = 0; b < S::V / S::RA; ++b) {
        const int j = t + b * S::NT, o = row_at<LGC>(j);
        cx<T> v[S::RA];
#pragma unroll
        for (int r = 0; r < S::RA; ++r) v[r] = s[o + r * S::MP];
        twiddle<T, LG, S::LGA, true>(v, j, tw);
        dft_n<T, S::RA, true>(v);
#pragma unroll
        for (int r = 0; r < S::RA; ++r) s[o + r * S::MP] = v[r];
    }
}

// ---------------------------------------------------------------------------
// Row pass
// ---------------------------------------------------------------------------

struct RowGeom {
    int lgh;        // log2(n1/2)
    int rows;       // rows per tile (a multiple of the rows of a warp)
    int64_t nrows;  // n2 n3
    int *err;       // device status word (bounded-wait time-outs)
    int *inject;    // failure-handling test hook (device word or null): when it
                    // holds 1 + this pass's kind (0 forward, 3 inverse), block 0
                    // clears it and issues no copies, so its bounded wait runs out
};

// What the node work of a row op sees: the tile's first row and node, its node
// count and the staged byte fields [kNB][nodes].
struct RowCtx {
    int64_t row0, p0;
    int nodes;
    const uint8_t *nb;
    __device__ __forceinline__ uchar2 b2(int k, int o) const
    {
        return *reinterpret_cast<const uchar2 *>(nb + k * nodes + o);
    }
};

// one copy of the transforms for the kernels that read the row length at run time
template <typename T, int LG, int LGC, bool INV>
__device__ __noinline__ void row_call(unsigned s, bool on, int t, const cx<T> *__restrict__ tw)
{
    if constexpr (INV)
        row_inverse<T, LG, LGC>(s, on, t, tw);
    else
        row_forward<T, LG, LGC>(s, on, t, tw);
}
template <typename T, int DIM, int LG, bool INV>
__device__ __forceinline__ void row_transform(int lgh, unsigned s, bool on, int t, const cx<T> *__restrict__ tw)
{
    constexpr bool D = sizeof(T) == 8;
    if constexpr (LG > 0) {
        if constexpr (INV)
            row_inverse<T, LG, row_lgc(D, DIM, LG)>(s, on, t, tw);
        else
            row_forward<T, LG, row_lgc(D, DIM, LG)>(s, on, t, tw);
    } else {
        switch (lgh) {
            case 4: row_call<T, 4, row_lgc(D, DIM, 4), INV>(s, on, t, tw); break;
            case 5: row_call<T, 5, row_lgc(D, DIM, 5), INV>(s, on, t, tw); break;
            case 6: row_call<T, 6, row_lgc(D, DIM, 6), INV>(s, on, t, tw); break;
            case 7: row_call<T, 7, row_lgc(D, DIM, 7), INV>(s, on, t, tw); break;
            case 8: row_call<T, 8, row_lgc(D, DIM, 8), INV>(s, on, t, tw); break;
            case 9: row_call<T, 9, row_lgc(D, DIM, 9), INV>(s, on, t, tw); break;
            default: row_call<T, 10, row_lgc(D, DIM, 10), INV>(s, on, t, tw); break;
        }
    }
}

// Block accumulator of a row op: Op::Acc when the op declares one, else DSum.
template <class Op, class = void>
struct op_acc {
    using type = DSum;
};
template <class Op>
struct op_acc<Op, std::void_t<typename Op::Acc>> {
    using type = typename Op::Acc;
};
// Ops that end with block reductions declare kReduce = true: they run on a
// bounded number of blocks, each walking several tiles, because every block
// writes its partial sums.
template <class Op, class = void>
struct op_reduce : std::false_type {
};
template <class Op>
struct op_reduce<Op, std::void_t<decltype(Op::kReduce)>> : std::bool_constant<Op::kReduce> {
};

// Ops with boundary-list work declare kEntries = true.
template <class Op, class = void>
struct op_entries : std::false_type {
};
template <class Op>
struct op_entries<Op, std::void_t<decltype(Op::kEntries)>> : std::bool_constant<Op::kEntries> {
};

// Ops that read fields of the plan's own (aligned) buffers after their inverse
// transforms name them for a prefetch to L2: kPre fields, pre(k). The CG's inverse
// pass reads p and r from memory, one tile at a time, with 17 warps on an SM to
// cover it (128^3 solve: 184 -> 182 ms).
template <class Op, class = void>
struct op_pre : std::integral_constant<int, 0> {
};
template <class Op>
struct op_pre<Op, std::void_t<decltype(Op::kPre)>> : std::integral_constant<int, Op::kPre> {
};

// Op interface:
//   static constexpr int kFin, kFout;  packed spectra read (inverse) / written (forward)
//   static constexpr int kNB;          byte fields bulk-copied for the tile's rows
//   const cx<T>* spec_in(int f); cx<T>* spec_out(int f);   row-major [row][n1/2]
//   const uint8_t* nb_src(int k);                          row-major [row][n1]
//   struct Nd; void load(Nd&, int64_t p0, int o): the global loads of the node
//        pair p0 + o, p0 + o + 1 (p0: first node of the tile); several pairs are
//        loaded before the first is used, and before the wait for the masks
//   void node2(ctx, o, nd, in0, in1, o0, o1, acc): nodes o and o + 1 of the tile;
//        in: kFin inverse-transformed values (unnormalised IDFT);
//        o: kFout values to transform
//   kEntries: const int *rows_off() (boundary-list offsets per row) and
//        void entry(int k, int64_t &p, T *s): node p of entry k and what it
//        adds to the kFin inverse-transformed values there. The entries of a
//        tile are worked off by all lanes at once between transform and node
//        work: looked up per node, the dependent loads of index, entry and
//        fields came one after the other in the lanes of boundary rows, and
//        those few blocks ran several times as long as the rest.
//   void block_done(acc): called by every thread at the end (block reductions)
// The masks of a tile arrive by bulk copy (one per byte field) behind a bounded
// wait, in the inverse passes while the transforms run.
// LG > 0: compiled for rows of 2^LG packed values (and the tile size launch_rows
// gives them): index arithmetic then is constants.
constexpr int kRowThreads = 384;
// Threads of a block and resident blocks the register allocation has to allow.
// Rows of up to 128 packed values: 64 registers a thread (FP64: 128); more warps
// then cover the copies (state-based 256 x 128 x 128: 254 -> 232 us, force at
// 256^3: 548 -> 538). Ops with reductions, whose accumulators spill then
// (128^3 solve: 184 -> 209 ms), and longer rows (1024 x 512 fracture steps: 1268 ->
// 1309 us) keep 80.
template <typename T, class Op, int LG>
constexpr int row_threads()
{
    constexpr int FB = Op::kFin > Op::kFout ? Op::kFin : Op::kFout;
    return LG > 0 ? 32 * row_warps(sizeof(T) == 8, 1 << LG, row_lgc(sizeof(T) == 8, Op::kDim, LG), FB) : kRowThreads;
}
template <typename T, class Op, int LG>
constexpr int row_blocks()
{
    if (LG == 0 || LG > 7 || op_reduce<Op>::value) return (sizeof(T) == 4 ? 768 : 384) / row_threads<T, Op, LG>();
    return (sizeof(T) == 4 ? 1024 : 512) / row_threads<T, Op, LG>();
}
template <typename T, class Op, int LG = 0>
__global__ void __launch_bounds__(row_threads<T, Op, LG>(), row_blocks<T, Op, LG>()) k_rows(RowGeom g, Op op, const cx<T> *__restrict__ tw)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    constexpr int FI = Op::kFin, FO = Op::kFout, NB = Op::kNB, FB = FI > FO ? FI : FO;
    const int lgh = LG > 0 ? LG : g.lgh;
    const int lgc = row_lgc(sizeof(T) == 8, Op::kDim, lgh);
    const int H = 1 << lgh, n1 = 2 * H, pitch = row_pitch(H, lgc);
    const int rows = LG > 0 ? row_tile_rows(sizeof(T) == 8, H, lgc, FB) : g.rows;
    unsigned long long *mbar = reinterpret_cast<unsigned long long *>(smem_raw);
    uint8_t *nb = smem_raw + 16;
    const unsigned spec_off = 16u + (unsigned)(NB * rows * n1);
    cx<T> *spec = reinterpret_cast<cx<T> *>(smem_raw + spec_off);
    const int tid = threadIdx.x;
    const int nt = row_lanes(H, lgc), tl = nt < 32 ? 32 : nt, wr = tl / nt;  // lanes of a row, of a task; its rows
    const int task0 = tid / tl, ntask = (int)blockDim.x / tl;
    auto at = [&](int e) { return e + (e >> lgc); };
    const int fstr = rows * pitch;  // field stride of the tile
    // node pairs loaded ahead: about 36 registers' worth
    constexpr int U0 = (int)(144 / sizeof(typename Op::Nd)), U = U0 < 1 ? 1 : U0 > 6 ? 6 : U0;
    const int lr = (tid & (tl - 1)) / nt, lt = tid & (nt - 1);
    const int groups = LG > 0 ? row_groups(sizeof(T) == 8, H, lgc, FB) : rows > wr ? rows / wr : 1;
    const int64_t ntiles = g.nrows / rows;
    constexpr bool kLoad = FI > 0 || NB > 0;
    if (kLoad && tid == 0) mbar_init(mbar, 1);
    pdl_wait();
    if constexpr (kLoad) __syncthreads();  // the barrier is initialised
    bool stall = false;
    if (kLoad && g.inject && blockIdx.x == 0 && tid == 0) {
        const int kind = FI > 0 ? 3 : 0;
        stall = atomicCAS(g.inject, kind + 1, 0) == kind + 1;
    }
    typename op_acc<Op>::type acc;
    unsigned phase = 0;
    for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        const int64_t row0 = tile * rows;
        // bulk copies of the tile: masks by one lane, spectra row by row by the
        // first warp
        if (kLoad && tid == 0 && !stall) {
            mbar_expect_tx(mbar, (unsigned)(NB * rows * n1 + FI * rows * H * (int)sizeof(cx<T>)));
#pragma unroll
            for (int k = 0; k < NB; ++k) bulk_load(nb + k * rows * n1, op.nb_src(k) + row0 * n1, rows * n1, mbar);
        }
        if constexpr (FI > 0) {
            if (tid < 32) {
                const bool skip = __shfl_sync(0xffffffffu, stall ? 1 : 0, 0) != 0;
                for (int i = tid; i < FI * rows && !skip; i += 32) {
                    const int f = i / rows, r = i - f * rows;
                    bulk_load(spec + (f * rows + r) * pitch, op.spec_in(f) + (row0 + r) * H,
                              (unsigned)(H * sizeof(cx<T>)), mbar);
                }
            }
        }
        if constexpr (op_pre<Op>::value > 0) {
            if (tid < op_pre<Op>::value)
                bulk_prefetch_l2(op.pre(tid) + row0 * n1, (unsigned)(rows * n1 * (int)sizeof(T)));
        }
        int k0 = 0, k1 = 0;
        if constexpr (op_entries<Op>::value) {
            k0 = op.rows_off()[row0];
            k1 = op.rows_off()[row0 + rows];
        }
        // false: the wait ran out
        auto arrive = [&]() {
            const bool ok = wait_for_copies(
                tid == 0, [&]() { return mbar_wait(mbar, phase, g.err); },
                [](bool x) { return __syncthreads_or(x) != 0; }, [&]() { mbar_drain(smem_u32(mbar), phase); });
            phase ^= 1u;
            return ok;
        };
        if constexpr (FI > 0) {
            if (!arrive()) return;
#pragma unroll 1
            for (int task = task0; task < FI * groups; task += ntask) {
                const int f = task / groups, r = (task - f * groups) * wr + lr;
                const unsigned s = spec_off + (unsigned)((f * rows + r) * pitch) * (unsigned)sizeof(cx<T>);
                const bool on = r < rows;
                row_transform<T, Op::kDim, LG, true>(lgh, s, LG > 0 || on, lt, tw);
            }
            __syncthreads();
        }
        if constexpr (op_entries<Op>::value) {
            if (k1 > k0) {
                T *base = reinterpret_cast<T *>(spec);
                for (int k = k0 + tid; k < k1; k += blockDim.x) {
                    int64_t p;
                    T s[FI];
                    op.entry(k, p, s);
                    const int nd = (int)(p - row0 * n1), rl = nd >> (lgh + 1), i1 = nd & (n1 - 1);
#pragma unroll
                    for (int f = 0; f < FI; ++f)
                        base[2 * ((f * rows + rl) * pitch + at(i1 >> 1)) + (i1 & 1)] += s[f];
                }
                __syncthreads();
            }
        }
        const RowCtx ctx{row0, row0 * n1, rows * n1, nb};
        const int pairs = rows * H, nthr = LG > 0 ? 32 * row_warps(sizeof(T) == 8, H, lgc, FB) : (int)blockDim.x;
        typename Op::Nd nd[U];
        auto load = [&](int i0) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int idx = i0 + u * nthr;
                if (idx < pairs) op.load(nd[u], ctx.p0, 2 * idx);
            }
        };
        if constexpr (FI == 0) load(tid);
        if constexpr (FI == 0 && NB > 0) {
            if (!arrive()) return;
        }
        for (int i0 = tid; i0 < pairs; i0 += U * nthr) {
            if (FI > 0 || i0 != tid) load(i0);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int idx = i0 + u * nthr;
                if (idx < pairs) {
                    cx<T> *sp = spec + (idx >> lgh) * pitch + at(idx & (H - 1));
                    T in0[FI > 0 ? FI : 1], in1[FI > 0 ? FI : 1], o0[FO > 0 ? FO : 1], o1[FO > 0 ? FO : 1];
#pragma unroll
                    for (int f = 0; f < FI; ++f) {
                        const cx<T> w = sp[f * fstr];
                        in0[f] = w.x;
                        in1[f] = w.y;
                    }
                    op.node2(ctx, 2 * idx, nd[u], in0, in1, o0, o1, acc);
#pragma unroll
                    for (int f = 0; f < FO; ++f) sp[f * fstr] = mk(o0[f], o1[f]);
                }
            }
        }
        if constexpr (FO > 0) {
            __syncthreads();
#pragma unroll 1
            for (int task = task0; task < FO * groups; task += ntask) {
                const int f = task / groups, r = (task - f * groups) * wr + lr;
                const unsigned s = spec_off + (unsigned)((f * rows + r) * pitch) * (unsigned)sizeof(cx<T>);
                const bool on = r < rows;
                row_transform<T, Op::kDim, LG, false>(lgh, s, LG > 0 || on, lt, tw);
                fence_proxy_async();
                if (nt > 32)
                    row_sync<64>();
                else
                    __syncwarp();
                if (lt == 0 && on) {
                    bulk_store(op.spec_out(f) + (row0 + r) * H, spec + (f * rows + r) * pitch,
                               (unsigned)(H * sizeof(cx<T>)));
                    bulk_commit();
                }
            }
            bulk_wait_read_all();  // shared memory is read before it is reused or given up
        }
        if (tile + gridDim.x < ntiles) {
            fence_proxy_async();  // the next tile's copies overwrite this one's data
            __syncthreads();
        }
    }
    op.block_done(acc);
}

}  // namespace pd

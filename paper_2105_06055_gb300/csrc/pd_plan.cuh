// Plan object and launch helpers of the GB300 FCBM-EC library (private).
#pragma once

#include <algorithm>
#include <utility>

#include <vector>

#include "pd_common.cuh"
#include "pd_cols.cuh"
#include "pd_fft.cuh"
#include "pd_rows.cuh"

namespace pd {

// One boundary node of the plan's G field (G != 0 only within delta of the
// body's boundary): the ncomp components in Sym order and the node index.
template <typename T>
struct GEntry {
    T g[6];
    int64_t p;
};

// Fields of a force evaluation of the nonlinear bond model: forward, inverse
// (the linearized models: one per component)
template <int D>
constexpr int kNLFwd = 2 * D + D * (D + 1) / 2;
template <int D>
constexpr int kNLInv = D + D * D + D * (D + 1) / 2 + D;

// Packed-spectrum slots of a plan in its own precision: what its widest pass
// touches, all of them in place. The nonlinear model's inverse fields; the
// linearized ones' adjoint (two vectors and the symmetric products), which holds the
// energy's fields and, in 3D, the state-based round's five slots.
constexpr int spec_slots_of(int dim, bool nonlinear)
{
    return nonlinear ? (dim == 2 ? kNLInv<2> : kNLInv<3>) : 2 * dim + dim * (dim + 1) / 2;
}
// Slots of one force evaluation without W; in FP64 on FP32 plans (the residual)
// there is nothing else.
constexpr int force_slots_of(int dim) { return dim == 2 ? 2 : 5; }

// Device-side view of the model used by the per-node and per-mode functors.
template <typename T>
struct Model {
    int dim;
    int n1, n2, n3;
    int h;             // n1 / 2
    int ky_half, kz_half;
    int64_t N;         // nodes
    int64_t nrows;     // n2 * n3
    const T *mhat;     // folded difference spectrum (K^(k) - K^(0)) / N, ncomp fields
    const T *ghat;     // folded dV/N * Σ g_i sin(theta) (state-based), 3 fields, or null
    int64_t fold_sz;   // entries per folded component: (h+1)(n2/2+1)(n3/2+1)
    const uint8_t *chi;
    const uint8_t *chi_om;  // d x N
    const T *G;        // ncomp x N boundary field for v = chi
    const GEntry<T> *gent;  // the same field as a list of boundary nodes, by row
    const int *goff;        // nrows + 1 offsets into gent
    const T *qt;       // 3 x N, state-based q_i(x) = dV (g_i * chi)
    const T *m3inv;    // N, 3/m(x) (0 outside the body)
    T ka;              // (3 kappa - 5 mu)/m0 (state-based)
};

struct HorizonDev {
    const int *off;   // 3 x cnt
    const double *c;  // ncomp x cnt: C_ij(xi) dV
    const double *g;  // 3 x cnt: g_i(xi) dV = omega xi_i dV (state-based), or
                      // a_i(xi) dV = alpha xi_i / |xi|^3 dV (nonlinear bond model)
    const double *w2; // cnt: omega |xi|^2 dV
    const double *cs; // cnt: c(xi) dV = alpha / |xi|^3 dV (nonlinear bond model), or null
    int cnt;
    int r[3];         // reach along each axis, in cells (the offsets' order is symmetric: bond
                      // cnt - 1 - c is opposite to bond c)
};

// Kernel-spectrum matrix of a mode from its table values (Sym order): the
// off-diagonal components along folded axes change sign
template <typename T>
__device__ __forceinline__ void load_mhat_s(int dim, const T *t, bool fy, bool fz, T *M /*3x3*/)
{
    if (dim == 2) {
        const T m11 = t[0], m22 = t[1], m12 = fy ? -t[2] : t[2];
        M[0] = m11; M[1] = m12; M[3] = m12; M[4] = m22;
    } else {
        const T m11 = t[0], m22 = t[1], m33 = t[2];
        const T m12 = fy ? -t[3] : t[3];
        const T m13 = fz ? -t[4] : t[4];
        const T m23 = (fy != fz) ? -t[5] : t[5];
        M[0] = m11; M[1] = m12; M[2] = m13;
        M[3] = m12; M[4] = m22; M[5] = m23;
        M[6] = m13; M[7] = m23; M[8] = m33;
    }
}

// gamma_i (odd in k_i) of a mode from its table values
template <typename T>
__device__ __forceinline__ void load_ghat_s(const T *t, bool fy, bool fz, T *g)
{
    g[0] = t[0];
    g[1] = fy ? -t[1] : t[1];
    g[2] = fz ? -t[2] : t[2];
}

}  // namespace pd

struct pd_plan {
    pd_problem prob;
    int dim, n1, n2, n3, h, ncomp;
    int64_t N, nrows;
    int lgl;            // log2 of the longest axis (twiddle tables of all lengths up to it)
    double dV, alpha;   // bond constant (or 30 mu / m0 for the state-based C)
    double ka, m0;      // state-based constants
    double lam_max;     // largest eigenvalue of the periodic symbol
    double wc = 0.0;    // critical energy density of bond breaking (problem Wc, or from s0)
    int state_based;    // model == PD_LIN_STATE && ka != 0 (dilatation round needed)
    int hcount;
    // device memory
    uint8_t *chi = nullptr, *chi_om = nullptr;
    uint8_t *mbits = nullptr;      // N: bit 0 chi_B, bit 1+c chi_Omega of component c
    int *hoff = nullptr;           // 3 x hcount integer offsets
    double *mhat64 = nullptr;      // ncomp x fold_sz
    float *mhat32 = nullptr;
    double *ghat64 = nullptr;      // 3 x fold_sz (state-based; nonlinear bond model: the a_i spectrum)
    double *chat64 = nullptr;      // fold_sz: (c^(k) - c^(0)) / N (nonlinear bond model)
    float *chat32 = nullptr;
    void *nlb = nullptr;           // nonlinear bond model: per boundary entry S(a_j, chi) (d values) and
                                   // S(c, chi) - c^(0) chi (slot 3), [ngent][4] in the plan's precision
    int nonlinear = 0;             // model == PD_NONLIN_BOND
    double body_count = 0.0;       // Σ chi
    float *ghat32 = nullptr;
    int64_t fold_sz = 0;
    double *G64 = nullptr;         // ncomp x N
    float *G32 = nullptr;
    // bond tables of the horizon sums on tiles (pd_horizon.cuh), null when the
    // horizon is too large for them
    float *hzt32 = nullptr;
    double *hzt64 = nullptr;
    int2 *hzcol = nullptr;
    int *goff = nullptr;           // nrows + 1: boundary-node list offsets per row
    int *gnode = nullptr;          // [ngent] node of each boundary entry (plane-pass cubes only)
    void *gpe = nullptr;           // [3][ngent] FP32 (G p) per boundary entry, written by the CG iteration
                                   // while its last-axis pass runs (plane-pass cubes only)
    void *gent64 = nullptr;        // GEntry<double>[ngent]
    void *gent32 = nullptr;        // GEntry<float>[ngent]
    // affine split of pd_force (pd_plan_set_affine_split): per boundary entry the
    // moments M_(ij)k = Σ_H chi(x+xi) C_ij(xi) dV o_k (o = integer offset), in the
    // plan's precision, [ngent][ncomp * dim]; the fitted coefficients; the body's
    // moment inverse and centre (host)
    void *aff_tab = nullptr;
    void *aff_coef = nullptr;      // 32 values of the plan's precision
    int affine_split = 0;
    int aff_ok = 0;                // body moments invertible
    int aff_c[3] = {0, 0, 0};      // centre node (integer grid indices)
    double aff_inv[16] = {};       // inverse of the (d+1)^2 normal matrix of the least-squares fit
    double aff_emax[3] = {0, 0, 0};
    int64_t ngent = 0;
    double *qt64 = nullptr, *m3inv64 = nullptr;  // state-based
    float *qt32 = nullptr, *m3inv32 = nullptr;
    pd::cx<double> *tw64 = nullptr;
    pd::cx<float> *tw32 = nullptr;
    void *spec32 = nullptr;        // spec32_slots x N floats (packed spectra)
    void *spec64 = nullptr;        // spec64_slots x N doubles
    int spec32_slots = 0, spec64_slots = 0;
    int *dev_status = nullptr;     // device status word (bounded-wait time-outs)
    int *inject = nullptr;         // row-pass stall word (pd_plan_inject_stall), next to dev_status
    void *work = nullptr;          // one allocation carved into the scratch fields below
    size_t work_bytes = 0;
    // scratch fields (plan precision T unless noted)
    void *cg_e = nullptr, *cg_r = nullptr, *cg_p = nullptr, *cg_q = nullptr;  // d x N each
    void *theta = nullptr;         // N, dilatation (state-based)
    void *Gw = nullptr;            // ncomp x N, boundary field of a node weight
    double *r64 = nullptr;         // d x N, FP64 residual / force
    double *theta64 = nullptr;     // N, FP64 dilatation for the FP64 residual
    double *red = nullptr;         // reduction partials and scalars
    int64_t bytes = 0;
    int64_t launches = 0;
    int nsm = 148;
    pd::HorizonDev hdev;  // device horizon tables (views into hoff)
    // per-pass timing (diagnostics): event pairs around each FFT-pass launch
    static constexpr int kEvPool = 1024;
    static constexpr int kKinds = 6;
    cudaEvent_t ev[2 * kEvPool] = {};
    int ev_kind[kEvPool] = {};
    int ev_used = 0;
    int ev_reserved = 0;            // pairs [0, ev_reserved) belong to captured graphs
    int prof_on = 0;                // bit k: time pass kind k
    int prof_cur = 0;               // the launch being bracketed is timed
    // cached CUDA graph of a chunk of CG iterations (per precision)
    cudaGraphExec_t cg_graph[2] = {nullptr, nullptr};
    int cg_graph_prof[2] = {0, 0};
    int cg_graph_ev[2][2] = {{0, 0}, {0, 0}};
    int64_t cg_graph_launches[2] = {0, 0};  // kernel launches per replay
    double *host_scal = nullptr;    // pinned host copy of the solver scalars
    cudaStream_t own_stream = nullptr;  // plan stream for captured work (never the legacy stream)
    cudaEvent_t ev_join[2] = {nullptr, nullptr};
    // second stream: (G p) per boundary entry beside the last-axis pass, for the CG's
    // inverse plane pass
    cudaStream_t aux_stream = nullptr;
    cudaEvent_t ev_fork[2] = {nullptr, nullptr};
    int no_fork = 0;  // set while capturing into conditional-node bodies (single stream there)
    int pdl = 1;      // pass kernels launched as programmatic dependents (griddepcontrol)
    // FP32 CG on cubes up to 128^3: halves of the iteration whose x1 and x2 transforms
    // run fused in plane passes (bit 0 forward, bit 1 inverse). By itself 1 on 32-node
    // planes (32^3: 32.1 us an iteration against 34.5 with row and column passes), 0 on
    // the larger ones (64^3: 38.3 against 41.4, 128^3: 108 against 122).
    int plane_passes = 0;
    double prof_ms[kKinds] = {};
    // tuning record (pd_plan_tuning): pd_plan_set_tuning's, or the passes' shapes as an
    // autotuner recorded them; the passes do not read it
    int tune_rows = 0;
    int tune_w[2] = {0, 0};
    int tune_sched = 0;
    int tune_stages = 0;
    int tune_stages_inv = 0;
    int energy_direct = 0; // pd_step_verlet: W by a direct horizon sum (pd_plan_set_energy_mode)
    int64_t prof_n[kKinds] = {};
};

namespace pd {

template <typename T>
Model<T> model_view(const pd_plan *p);

template <typename T>
inline T *spec_buf(const pd_plan *p);
template <>
inline float *spec_buf<float>(const pd_plan *p) { return (float *)p->spec32; }
template <>
inline double *spec_buf<double>(const pd_plan *p) { return (double *)p->spec64; }

template <typename T>
inline const cx<T> *tw_buf(const pd_plan *p);
template <>
inline const cx<float> *tw_buf<float>(const pd_plan *p) { return p->tw32; }
template <>
inline const cx<double> *tw_buf<double>(const pd_plan *p) { return p->tw64; }

pd_status set_smem_attr(const void *func, size_t smem);

// pass kinds for the timing facility
enum PassKind { PASS_ROWS_FWD = 0, PASS_COLS = 1, PASS_LAST = 2, PASS_ROWS_INV = 3, PASS_PLANE_FWD = 4, PASS_PLANE_INV = 5 };
pd_status prof_harvest(pd_plan *p);
pd_status prof_harvest_range(pd_plan *p, int b, int e);

// Layout of the plan's FP64 reduction buffer (65536 doubles).
constexpr int kRedPart = 0;       // block partial sums (up to kMaxPart)
constexpr int kMaxPart = 58000;
constexpr int kRedScal = 60000;   // solver scalars
constexpr int kRedVerlet = 62000; // Verlet counters
// the device status word sits in the last 64 bytes
// Events recorded while the stream is being captured must become external
// event nodes of the graph, so that each replay records them.
inline cudaError_t prof_record(cudaEvent_t e, cudaStream_t st)
{
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    cudaError_t r = cudaStreamIsCapturing(st, &cs);
    if (r != cudaSuccess) return r;
    return cs == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(e, st, cudaEventRecordExternal)
                                               : cudaEventRecord(e, st);
}

inline pd_status prof_begin(pd_plan *p, int kind, cudaStream_t st)
{
    p->prof_cur = ((p->prof_on >> kind) & 1) != 0;
    if (!p->prof_cur) return PD_OK;
    if (p->ev_used == pd_plan::kEvPool) PD_TRY(prof_harvest(p));
    if (p->ev_used == pd_plan::kEvPool) {
        set_error("profiling event pool exhausted");
        return PD_ERR_ARG;
    }
    p->ev_kind[p->ev_used] = kind;
    PD_CUDA_TRY(prof_record(p->ev[2 * p->ev_used], st));
    return PD_OK;
}
inline pd_status prof_end(pd_plan *p, cudaStream_t st)
{
    if (!p->prof_cur) return PD_OK;
    PD_CUDA_TRY(prof_record(p->ev[2 * p->ev_used + 1], st));
    p->ev_used++;
    return PD_OK;
}

// Launch with the programmatic-stream-serialization attribute when pdl is set:
// the kernel may start while its predecessor in the stream finishes and waits
// for it with griddepcontrol.wait (every pass kernel does, before it touches
// data of the preceding pass).
template <typename... KArgs, typename... Args>
inline pd_status launch_k(bool pdl, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                          Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl ? attr : nullptr;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    if (e != cudaSuccess) {
        set_error("kernel launch failed: %s", cudaGetErrorString(e));
        return PD_ERR_CUDA;
    }
    return PD_OK;
}

// Row kernels are compiled per row length, with the index arithmetic as
// constants (at 128^3 the forward pass: 28 us with the length read at run time, 16
// us so), for boxes of 64 to 2048 nodes along x1 in 2D and 32 to 512 in 3D; the
// remaining lengths share one kernel that reads it.
template <typename T, class Op>
auto rows_kernel(int lgh)
{
    using K = decltype(&k_rows<T, Op>);
    if constexpr (Op::kDim == 2) {
        switch (lgh) {
            case 9: return (K)&k_rows<T, Op, 9>;
            case 10: return (K)&k_rows<T, Op, 10>;
            default: break;
        }
    } else if (lgh == 4) {
        return (K)&k_rows<T, Op, 4>;
    }
    switch (lgh) {
        case 5: return (K)&k_rows<T, Op, 5>;
        case 6: return (K)&k_rows<T, Op, 6>;
        case 7: return (K)&k_rows<T, Op, 7>;
        case 8: return (K)&k_rows<T, Op, 8>;
        default: break;
    }
    return (K)&k_rows<T, Op>;
}

// Rows per tile of a row pass over `fields` fields: row_tile_rows, fewer when the grid
// has fewer (*whole: the tile size the fixed-length kernels are compiled for).
template <typename T, int D>
int row_tile(const pd_plan *p, int fields, bool *whole)
{
    int rows = row_tile_rows(sizeof(T) == 8, p->h, row_lgc(sizeof(T) == 8, D, ilog2(p->h)), fields);
    *whole = p->nrows % rows == 0;
    while (p->nrows % rows) rows >>= 1;
    return rows;
}

// Row pass: tile by row_tile, warps by row_warps. Passes with block reductions run on at most 8 blocks per SM
// (each block writes partial sums), all with as many tiles as far as it goes; the
// others on a block per tile. *grid_out
// receives the block count.
template <typename T, class Op>
pd_status launch_rows(pd_plan *p, const Op &op, cudaStream_t st, unsigned *grid_out = nullptr)
{
    constexpr int FB = Op::kFin > Op::kFout ? Op::kFin : Op::kFout;
    RowGeom g;
    g.lgh = ilog2(p->h);
    const int lgc = row_lgc(sizeof(T) == 8, Op::kDim, g.lgh);
    bool whole = true;
    g.rows = row_tile<T, Op::kDim>(p, FB, &whole);
    g.nrows = p->nrows;
    g.err = p->dev_status;
    g.inject = p->inject;
    const size_t smem =
        16 + (size_t)Op::kNB * g.rows * p->n1 + (size_t)FB * g.rows * row_pitch(p->h, lgc) * sizeof(cx<T>);
    int64_t grid = p->nrows / g.rows;
    if (op_reduce<Op>::value) {
        const int64_t per = (grid + 8 * (int64_t)p->nsm - 1) / (8 * (int64_t)p->nsm);  // tiles a block
        grid = (grid + per - 1) / per;
    }
    if (grid_out) *grid_out = (unsigned)grid;
    const auto kern = whole ? rows_kernel<T, Op>(g.lgh) : &k_rows<T, Op>;
    PD_TRY(set_smem_attr((const void *)kern, smem));
    PD_TRY(prof_begin(p, Op::kFin > 0 ? PASS_ROWS_INV : PASS_ROWS_FWD, st));
    PD_TRY(launch_k(p->pdl != 0, kern, dim3((unsigned)grid), dim3(32 * row_warps(sizeof(T) == 8, p->h, lgc, FB)), smem,
                    st, g, op, tw_buf<T>(p)));
    PD_TRY(prof_end(p, st));
    p->launches++;
    return PD_OK;
}

template <typename T>
inline int spec_slots(const pd_plan *p) { return sizeof(T) == 8 ? p->spec64_slots : p->spec32_slots; }

// PD_ERR_ARG unless the plan has the slots below n (every pipeline asks before its first
// pass writes them).
template <typename T>
pd_status check_slots(const pd_plan *p, int n)
{
    if (n <= spec_slots<T>(p)) return PD_OK;
    set_error("a pass over %d spectra on a plan with %d", n, spec_slots<T>(p));
    return PD_ERR_ARG;
}

// Geometry of a column pass along x2 (zaxis 0) or x3 (zaxis 1).
template <typename T>
inline ColArgs<T> col_args(const pd_plan *p, int zaxis)
{
    ColArgs<T> g;
    g.spec = reinterpret_cast<cx<T> *>(const_cast<T *>(spec_buf<T>(p)));
    g.fs = p->N / 2;
    g.ls = zaxis ? (int64_t)p->n2 * p->h : (int64_t)p->h;
    g.os = (int64_t)p->n2 * p->h;
    g.lgh = ilog2(p->h);
    g.n2 = zaxis ? p->n2 : 1;
    g.nspec = 0;
    g.sw = 0;
    g.zaxis = zaxis;
    return g;
}

template <typename T, int LG, bool INV>
pd_status launch_plain(pd_plan *p, int slot0, int fields, cudaStream_t st)
{
    using S = PlainShape<T, LG, INV>;
    const auto kern = k_col_plain<T, LG, INV>;
    PD_TRY(set_smem_attr((const void *)kern, S::smem));
    return launch_k(p->pdl != 0, kern, dim3((unsigned)(p->h / S::W), (unsigned)p->n3, (unsigned)fields),
                    dim3(S::THREADS), S::smem, st, col_args<T>(p, 0), slot0, tw_buf<T>(p));
}

// Plain transforms along x2 of the spectra in slots slot0 ... slot0 + fields - 1, in place.
template <typename T>
pd_status col_pass(pd_plan *p, int slot0, int fields, bool inverse, cudaStream_t st);

template <typename T, class Op, int LG>
pd_status launch_comb_lg(pd_plan *p, const Op &op, cudaStream_t st)
{
    using S = CombShape<T, Op, LG>;
    const auto kern = k_col_comb<T, Op, LG>;
    PD_TRY(set_smem_attr((const void *)kern, S::smem));
    const int z = p->dim == 3 ? 1 : 0;
    ColArgs<T> g = col_args<T>(p, z);
    const unsigned tiles = (unsigned)((int64_t)(z ? p->n2 : 1) * p->h / S::W);
    // pairs of kx = 0 columns: k2 = 0 ... n2/2 in 3D, one column in 2D
    g.sw = z ? special_cols(LG, S::W, tiles, p->nsm) : special_cols(0, S::W, 0, 0);
    g.nspec = ((z ? p->n2 + 2 : 2) + g.sw - 1) / g.sw;
    return launch_k(p->pdl != 0, kern, dim3(tiles + (unsigned)g.nspec), dim3(S::THREADS), S::smem, st, g, op,
                    tw_buf<T>(p));
}

// The last-axis pass: forward transform, spectral combine, inverse transform.
template <typename T, class Op>
pd_status launch_comb(pd_plan *p, const Op &op, cudaStream_t st)
{
    PD_TRY(prof_begin(p, PASS_LAST, st));
    pd_status s = PD_ERR_SIZE;
    switch (ilog2(p->dim == 3 ? p->n3 : p->n2)) {
        case 4: s = launch_comb_lg<T, Op, 4>(p, op, st); break;
        case 5: s = launch_comb_lg<T, Op, 5>(p, op, st); break;
        case 6: s = launch_comb_lg<T, Op, 6>(p, op, st); break;
        case 7: s = launch_comb_lg<T, Op, 7>(p, op, st); break;
        case 8: s = launch_comb_lg<T, Op, 8>(p, op, st); break;
        case 9: s = launch_comb_lg<T, Op, 9>(p, op, st); break;
        case 10: s = launch_comb_lg<T, Op, 10>(p, op, st); break;
        default: set_error("axis length outside 16..1024"); break;
    }
    PD_TRY(s);
    PD_TRY(prof_end(p, st));
    p->launches++;
    return PD_OK;
}

}  // namespace pd

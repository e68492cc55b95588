// Autotuner: picks, for the static solver on FP32 cubes up to 128^3, whether the
// forward half of the CG iteration runs as a plane pass, by timing a chunk of CG
// iterations (pd_plan_autotune_solve) on the plan's own workspace with CUDA
// events.
//
// The tile shapes of the row and column passes are compile-time constants per
// axis length (pd_rows.cuh, pd_cols.cuh): with the length and the shape known
// the index arithmetic folds away, which gained more than any choice of shape
// at run time did. The tuning record (pd_plan_tuning) keeps its six entries: what
// pd_plan_set_tuning stored, or, from an autotuner on, the shapes the passes of the
// plan's force evaluation run with.
#include "pd_plan.cuh"

using namespace pd;

struct pd_batch;
extern "C" pd_plan *pd_batch_plan(pd_batch *B, int i);
extern "C" int pd_batch_size(const pd_batch *B);

namespace pd {
pd_status time_cg_chunk(pd_plan *p, cudaEvent_t e0, cudaEvent_t e1, float *ms_out);
}

namespace {

void drop_graphs(pd_plan *p)
{
    for (int k = 0; k < 2; ++k)
        if (p->cg_graph[k]) {
            cudaGraphExecDestroy(p->cg_graph[k]);
            p->cg_graph[k] = nullptr;
        }
}

// Tile widths (columns) of the x2 pass and of the last-axis pass over FB fields.
template <typename T>
int x2_width(int lg)
{
    switch (lg) {
        case 4: return PlainShape<T, 4, false>::W;
        case 5: return PlainShape<T, 5, false>::W;
        case 6: return PlainShape<T, 6, false>::W;
        case 7: return PlainShape<T, 7, false>::W;
        case 8: return PlainShape<T, 8, false>::W;
        case 9: return PlainShape<T, 9, false>::W;
        default: return PlainShape<T, 10, false>::W;
    }
}
template <int D, int FB>
struct Fields {
    static constexpr int kFin = FB, kFout = FB, kDim = D;
};
template <typename T, class F>
int last_width(int lg)
{
    switch (lg) {
        case 4: return CombShape<T, F, 4>::W;
        case 5: return CombShape<T, F, 5>::W;
        case 6: return CombShape<T, F, 6>::W;
        case 7: return CombShape<T, F, 7>::W;
        case 8: return CombShape<T, F, 8>::W;
        case 9: return CombShape<T, F, 9>::W;
        default: return CombShape<T, F, 10>::W;
    }
}

// The tuning record of the plan's force evaluation (without W): rows per tile of the
// forward row pass, tile widths, one schedule, one tile at a time in the row passes.
template <typename T, int D>
void record_shapes(pd_plan *p)
{
    bool whole = true;
    p->tune_rows = row_tile<T, D>(p, p->nonlinear ? kNLFwd<D> : D, &whole);
    p->tune_w[0] = D == 3 ? x2_width<T>(ilog2(p->n2)) : 0;
    const int lg = ilog2(D == 3 ? p->n3 : p->n2);
    p->tune_w[1] = p->nonlinear ? last_width<T, Fields<D, kNLInv<D>>>(lg) : last_width<T, Fields<D, D>>(lg);
    p->tune_sched = 0;
    p->tune_stages = p->tune_stages_inv = 1;
}
void record_shapes(pd_plan *p)
{
    if (p->prob.fp64)
        p->dim == 2 ? record_shapes<double, 2>(p) : record_shapes<double, 3>(p);
    else
        p->dim == 2 ? record_shapes<float, 2>(p) : record_shapes<float, 3>(p);
}

// target 1: the static solver's CG iteration, 0: force evaluations (nothing to choose)
pd_status tune_plan(pd_plan *p, cudaStream_t caller, int target = 0)
{
    // the inverse plane pass is not a candidate: a lone chunk timed it faster,
    // whole solves slower (128^3: 115.3 against 105.9 ms per solve)
    if (target == 1 && p->dim == 3 && !p->prob.fp64 && !p->state_based && p->n1 == p->n2 &&
        (p->n1 == 32 || p->n1 == 64 || p->n1 == 128)) {
        PD_CUDA_TRY(cudaEventRecord(p->ev_join[0], caller));
        PD_CUDA_TRY(cudaStreamWaitEvent(p->own_stream, p->ev_join[0], 0));
        const int prof = p->prof_on;
        p->prof_on = 0;
        cudaEvent_t e0 = nullptr, e1 = nullptr;
        PD_CUDA_TRY(cudaEventCreate(&e0));
        PD_CUDA_TRY(cudaEventCreate(&e1));
        pd_status s = PD_OK;
        float tbest = 1e30f;
        int best = p->plane_passes;
        for (int c : {1, 0}) {
            if (s != PD_OK) break;
            p->plane_passes = c;
            drop_graphs(p);
            float ms = 0.f;
            s = time_cg_chunk(p, e0, e1, &ms);
            if (s == PD_OK && ms < tbest) {
                tbest = ms;
                best = c;
            }
        }
        p->plane_passes = best;
        p->prof_on = prof;
        drop_graphs(p);
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        if (s != PD_OK) return s;
        PD_CUDA_TRY(cudaEventRecord(p->ev_join[1], p->own_stream));
        PD_CUDA_TRY(cudaStreamWaitEvent(caller, p->ev_join[1], 0));
    }
    record_shapes(p);
    return PD_OK;
}

}  // namespace

extern "C" pd_status pd_plan_autotune(pd_plan *p, void *stream)
{
    if (!p) {
        set_error("pd_plan_autotune: null plan");
        return PD_ERR_ARG;
    }
    return tune_plan(p, (cudaStream_t)stream);
}

extern "C" pd_status pd_plan_autotune_solve(pd_plan *p, void *stream)
{
    if (!p) {
        set_error("pd_plan_autotune_solve: null plan");
        return PD_ERR_ARG;
    }
    if (p->nonlinear) {
        set_error("pd_plan_autotune_solve: the nonlinear bond model is available through pd_force only");
        return PD_ERR_ARG;
    }

    return tune_plan(p, (cudaStream_t)stream, 1);
}

extern "C" pd_status pd_plan_tuning(const pd_plan *p, int *out6)
{
    if (!p || !out6) {
        set_error("pd_plan_tuning: null argument");
        return PD_ERR_ARG;
    }
    out6[0] = p->tune_rows;
    out6[1] = p->tune_w[0];
    out6[2] = p->tune_w[1];
    out6[3] = p->tune_sched;
    out6[4] = p->tune_stages;
    out6[5] = p->tune_stages_inv;
    return PD_OK;
}

extern "C" pd_status pd_batch_autotune(pd_batch *B, void *stream)
{
    if (!B) {
        set_error("pd_batch_autotune: null batch");
        return PD_ERR_ARG;
    }
    for (int i = 0; i < pd_batch_size(B); ++i) PD_TRY(tune_plan(pd_batch_plan(B, i), (cudaStream_t)stream));
    return PD_OK;
}

extern "C" pd_status pd_plan_set_plane_passes(pd_plan *p, int on)
{
    if (!p || on < 0 || on > 3) {
        set_error("pd_plan_set_plane_passes: null plan or mask not in 0..3");
        return PD_ERR_ARG;
    }
    p->plane_passes = on;
    drop_graphs(p);
    return PD_OK;
}

extern "C" pd_status pd_plan_set_tuning(pd_plan *p, const int *in6)
{
    if (!p || !in6) {
        set_error("pd_plan_set_tuning: null argument");
        return PD_ERR_ARG;
    }
    const int r = in6[0], wx = in6[1], wl = in6[2], sc = in6[3], ns = in6[4], ni = in6[5];
    auto pow2_or_zero = [](int v) { return v == 0 || (v > 0 && (v & (v - 1)) == 0); };
    // (a column tile is at least a pair of columns wide)
    if (!pow2_or_zero(r) || r > 256 || !pow2_or_zero(wx) || wx == 1 || wx > 32 || !pow2_or_zero(wl) || wl == 1 ||
        wl > 32 || (sc != 0 && sc != 1) || ns < 0 || ns > 2 || ni < 0 || ni > 2) {
        set_error("pd_plan_set_tuning: rows and widths must be 0 or powers of two (rows <= 256, widths 2..32), "
                  "schedule 0 or 1, stages 0, 1 or 2");
        return PD_ERR_ARG;
    }
    p->tune_rows = r;
    p->tune_w[0] = wx;
    p->tune_w[1] = wl;
    p->tune_sched = sc;
    p->tune_stages = ns;
    p->tune_stages_inv = ni;
    return PD_OK;
}

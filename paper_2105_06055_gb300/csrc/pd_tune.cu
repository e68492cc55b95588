// Autotuner: picks, for the static solver on FP32 cubes up to 128^3, whether the
// forward half of the CG iteration runs as a plane pass, by timing a chunk of CG
// iterations (pd_plan_autotune_solve) on the plan's own workspace with CUDA
// events.
//
// The tile shapes of the row and column passes are compile-time constants per
// axis length (pd_rows.cuh, pd_cols.cuh): with the length and the shape known
// the index arithmetic folds away, which gained more than any choice of shape
// at run time did. The tuning record (pd_plan_tuning, pd_plan_set_tuning) keeps
// its six entries; autotuning reports the nominal shape in those that are 0.
#include <map>
#include <tuple>

#include "pd_plan.cuh"

using namespace pd;

struct pd_batch;
void pd_batch_invalidate(pd_batch *B);
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
    if (!p->tune_rows) p->tune_rows = row_warp_rows(p->h, row_lgc(p->prob.fp64 != 0, p->dim, ilog2(p->h)));
    for (int k = 0; k < 2; ++k)
        if (!p->tune_w[k]) p->tune_w[k] = p->prob.fp64 ? 8 : 16;
    if (!p->tune_stages) p->tune_stages = 1;
    if (!p->tune_stages_inv) p->tune_stages_inv = 1;
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
    // one search per distinct grid / precision / operator; the others copy it
    std::map<std::tuple<int, int, int, int, int, int>, pd_plan *> done;
    for (int i = 0; i < pd_batch_size(B); ++i) {
        pd_plan *p = pd_batch_plan(B, i);
        const auto key = std::make_tuple(p->dim, p->n1, p->n2, p->n3, p->prob.fp64, p->state_based);
        auto it = done.find(key);
        if (it == done.end()) {
            PD_TRY(tune_plan(p, (cudaStream_t)stream));
            done[key] = p;
        } else {
            p->tune_rows = it->second->tune_rows;
            p->tune_w[0] = it->second->tune_w[0];
            p->tune_w[1] = it->second->tune_w[1];
            p->tune_sched = it->second->tune_sched;
            p->tune_stages = it->second->tune_stages;
            p->tune_stages_inv = it->second->tune_stages_inv;
            drop_graphs(p);
        }
    }
    pd_batch_invalidate(B);
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
    // a column tile is at least 2 complex values wide: its first column, and so the
    // x coordinate of every tensor copy, is then a multiple of 16 bytes
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
    drop_graphs(p);
    return PD_OK;
}

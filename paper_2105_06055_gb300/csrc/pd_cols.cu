// The plain x2 column passes (one unit, every length and precision).
#include "pd_plan.cuh"

namespace pd {

template <typename T>
pd_status col_pass(pd_plan *p, int slot0, int fields, bool inverse, cudaStream_t st)
{
    PD_TRY(prof_begin(p, PASS_COLS, st));
    pd_status s = PD_ERR_SIZE;
#define PD_COL_CASE(LG)                                                          \
    case LG:                                                                     \
        s = inverse ? launch_plain<T, LG, true>(p, slot0, fields, st)            \
                    : launch_plain<T, LG, false>(p, slot0, fields, st);          \
        break;
    switch (ilog2(p->n2)) {
        PD_COL_CASE(4)
        PD_COL_CASE(5)
        PD_COL_CASE(6)
        PD_COL_CASE(7)
        PD_COL_CASE(8)
        PD_COL_CASE(9)
        PD_COL_CASE(10)
        default: set_error("axis length outside 16..1024"); break;
    }
#undef PD_COL_CASE
    PD_TRY(s);
    PD_TRY(prof_end(p, st));
    p->launches++;
    return PD_OK;
}
template pd_status col_pass<float>(pd_plan *, int, int, bool, cudaStream_t);
template pd_status col_pass<double>(pd_plan *, int, int, bool, cudaStream_t);

}  // namespace pd

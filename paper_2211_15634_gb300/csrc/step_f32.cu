// FP32 forward step dispatch (deviation storage D = T - T_ref): TMA z-march when nx is a
// multiple of 4, else its row-by-row form (zrag_tile.cuh; the two-float state zcomp_rag.cu) below
// 2^31 nodes, else the plain column march.  Small grids take the column march (stencil_basic.cuh): on aligned
// rows inside a time loop only, on other rows a single step too.
#include "internal.h"
#include "stencil_basic.cuh"
#include "zmarch.h"

namespace psd {

static CoefT<float> coef_f32(StepCoef c) {
    return CoefT<float>{(float)c.dtlam, (float)c.ax, (float)c.ay, (float)c.az};
}

cudaError_t launch_step_f32(float *T2, const float *T, const float *Ci, StepCoef c, Grid3 g,
                            cudaStream_t s, bool write_bnd, bool in_loop) {
    if (step_small(g, Z_F32, in_loop))
        return launch_step_basic<float, false>(T2, T, nullptr, nullptr, Ci, coef_f32(c), g, s, true);
    if (step_tma_ok(g, 4, T2, T, Ci))
        return launch_zmarch(Z_F32, T2, T, nullptr, nullptr, Ci, c, g, s, write_bnd);
    if (step_ragged_ok(g, 4, T2, T, Ci))
        return launch_zmarch_ragged(Z_F32, T2, T, Ci, c, g, s, write_bnd);
    return launch_step_basic<float, false>(T2, T, nullptr, nullptr, Ci, coef_f32(c), g, s, false);
}

// Two-float state (D, E) -> (D2, E2): the TMA z-march stages E like T (odd rows: zcomp_rag.cu).
cudaError_t launch_step_f32_comp(float *T2, const float *T, float *E2, const float *E, const float *Ci,
                                 StepCoef c, Grid3 g, cudaStream_t s, bool in_loop) {
    if (step_small(g, Z_F32_COMP, in_loop))
        return launch_step_basic<float, true>(T2, T, E2, E, Ci, coef_f32(c), g, s, true);
    if (step_tma_ok(g, 4, T2, T, Ci) && step_tma_ok(g, 4, E2, E, Ci))
        return launch_zmarch(Z_F32_COMP, T2, T, E2, E, Ci, c, g, s);
    if (comp_ragged_ok(g, T2, T, Ci))
        return launch_comp_ragged(T2, T, E2, E, Ci, c, g, s);
    return launch_step_basic<float, true>(T2, T, E2, E, Ci, coef_f32(c), g, s, false);
}

const char *step_f32_kernel_name(Grid3 g, const void *T2, const void *T, const void *Ci) {
    if (step_small(g, Z_F32, false)) return "k_step_basic<float>";
    if (step_tma_ok(g, 4, T2, T, Ci)) return "k_zmarch<F32>";
    return step_ragged_ok(g, 4, T2, T, Ci) ? "k_zmarch_rag<F32>" : "k_step_basic<float>";
}

}  // namespace psd

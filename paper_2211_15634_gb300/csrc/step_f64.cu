// FP64 forward step dispatch.
//   fast:   TMA z-march with one-DFMA emulated arithmetic (even nx), its row-by-row form
//           (odd nx below 2^31 nodes, spacings within 16 of each other), else the plain
//           column march with the same arithmetic.  Small grids take the column march
//           (stencil_basic.cuh): even nx inside a time loop only (and not Ci as given on equal
//           spacings), odd nx a single step too.
//   native: plain column march with ordinary FP64 instructions.
#include "internal.h"
#include "stencil_basic.cuh"
#include "zmarch.h"

namespace psd {

static CoefT<double> coef_f64(StepCoef c) { return CoefT<double>{c.dtlam, c.ax, c.ay, c.az}; }

cudaError_t launch_step_f64_native(double *T2, const double *T, const double *Ci, StepCoef c,
                                   Grid3 g, cudaStream_t s) {
    return launch_step_basic<double, false>(T2, T, nullptr, nullptr, Ci, coef_f64(c), g, s, false);
}

bool emu_ok(StepCoef c) {
    const double k[3] = {c.dtlam * c.ax, c.dtlam * c.ay, c.dtlam * c.az};
    for (double v : k)
        if (!(v > 2.2250738585072014e-308 && v < 1e300)) return false;  // positive normal
    return true;
}

cudaError_t launch_step_f64_fast(double *T2, const double *T, const double *Ci, StepCoef c,
                                 Grid3 g, cudaStream_t s, bool write_bnd, bool in_loop) {
    if (!emu_ok(c)) return launch_step_f64_native(T2, T, Ci, c, g, s);
    const bool iso = c.ax == c.ay && c.ay == c.az;
    const EmuCoef ek = emu_coef(c.dtlam, c.ax, c.ay, c.az);
    if (step_small(g, iso ? Z_F64_EMU_ISO : Z_F64_EMU_ANISO, in_loop))
        return launch_step_basic_emu(T2, T, Ci, ek, iso, g, s, false, true);
    if (step_tma_ok(g, 8, T2, T, Ci))
        return launch_zmarch(iso ? Z_F64_EMU_ISO : Z_F64_EMU_ANISO, T2, T, nullptr, nullptr, Ci, c, g, s,
                             write_bnd);
    if (ek.axes != AX_FAR && step_ragged_ok(g, 8, T2, T, Ci))
        return launch_zmarch_ragged(iso ? Z_F64_EMU_ISO : Z_F64_EMU_ANISO, T2, T, Ci, c, g, s, write_bnd);
    return launch_step_basic_emu(T2, T, Ci, ek, iso, g, s, false, false);
}

// Ci already scaled to dt*lam*_dx^2*Ci (isotropic grids): one DFMA per node.
cudaError_t launch_step_f64_scaled(double *T2, const double *T, const double *Cs, Grid3 g,
                                   cudaStream_t s, bool write_bnd, bool in_loop) {
    const StepCoef dummy{1.0, 1.0, 1.0, 1.0};
    const EmuCoef ek{};
    if (step_small(g, Z_F64_SCALED, in_loop)) return launch_step_basic_emu(T2, T, Cs, ek, true, g, s, true, true);
    if (step_tma_ok(g, 8, T2, T, Cs))
        return launch_zmarch(Z_F64_SCALED, T2, T, nullptr, nullptr, Cs, dummy, g, s, write_bnd);
    if (step_ragged_ok(g, 8, T2, T, Cs))
        return launch_zmarch_ragged(Z_F64_SCALED, T2, T, Cs, dummy, g, s, write_bnd);
    return launch_step_basic_emu(T2, T, Cs, ek, true, g, s, true, false);
}

bool step_takes_march(int dtype, bool scaled, bool native, bool in_loop, StepCoef c, Grid3 g, const void *T2,
                      const void *T, const void *Ci) {
    auto march = [&](int esz) { return step_tma_ok(g, esz, T2, T, Ci) || step_ragged_ok(g, esz, T2, T, Ci); };
    if (dtype != PS_F64) return !step_small(g, Z_F32, in_loop) && march(4);  // launch_step_f32
    if (scaled) return !step_small(g, Z_F64_SCALED, in_loop) && march(8);    // launch_step_f64_scaled
    if (native || !emu_ok(c)) return false;                                       // the column kernel
    const bool iso = c.ax == c.ay && c.ay == c.az;                                // launch_step_f64_fast
    if (step_small(g, iso ? Z_F64_EMU_ISO : Z_F64_EMU_ANISO, in_loop)) return false;
    return step_tma_ok(g, 8, T2, T, Ci) ||
           (emu_coef(c.dtlam, c.ax, c.ay, c.az).axes != AX_FAR && step_ragged_ok(g, 8, T2, T, Ci));
}

const char *step_f64_kernel_name(Grid3 g, const void *T2, const void *T, const void *Ci, StepCoef c,
                                 bool scaled) {
    if (scaled) {
        if (step_small(g, Z_F64_SCALED, false)) return "k_step_basic_emu";
        if (step_ragged_ok(g, 8, T2, T, Ci)) return "k_zmarch_rag<F64_SCALED>";
        if (!step_tma_ok(g, 8, T2, T, Ci)) return "k_step_basic_emu";
        return f64_scaled_wide(g, T2, T, Ci) ? "k_zmarch<F64_SCALED4>" : "k_zmarch<F64_SCALED>";
    }
    if (!emu_ok(c)) return "k_step_basic<double>";
    const bool iso = c.ax == c.ay && c.ay == c.az;
    if (step_small(g, iso ? Z_F64_EMU_ISO : Z_F64_EMU_ANISO, false)) return "k_step_basic_emu";
    if (step_tma_ok(g, 8, T2, T, Ci)) return iso ? "k_zmarch<F64_EMU_ISO>" : "k_zmarch<F64_EMU_ANISO>";
    if (emu_coef(c.dtlam, c.ax, c.ay, c.az).axes != AX_FAR && step_ragged_ok(g, 8, T2, T, Ci))
        return iso ? "k_zmarch_rag<F64_EMU_ISO>" : "k_zmarch_rag<F64_EMU_ANISO>";
    return "k_step_basic_emu";
}

}  // namespace psd

// Declarations of the TMA-fed z-march step kernels (zmarch.cu).
#pragma once

#include <cuda.h>

#include "emu64.cuh"
#include "internal.h"

namespace psd {

enum ZMode {
    Z_F64_EMU_ISO = 0,       // one DFMA per node, 64x64 high multiply by K
    Z_F64_EMU_ANISO = 1,     // as above, the axes' K as integers at one exponent
    Z_F64_NATIVE = 2,        // plain FP64 instructions
    Z_F32 = 3,
    Z_F32_COMP = 4,
    Z_F64_EMU_ISO_DMUL = 5,  // two FP64 ops per node: fma(Ci*K, S, T)
    Z_F64_SCALED = 6,        // Ci already holds dt*lam*_d^2*Ci: fma(Cs, S, T)
    Z_F64_SCALED4 = 7,       // as Z_F64_SCALED, four nodes per thread (32-byte accesses)
    Z_F64_EMU_ANISO4 = 9,    // as Z_F64_EMU_ANISO, four nodes per thread
    Z_F64_EMU_ANISO_SPREAD = 10,  // spacings up to 16 apart (AX_SPREAD)
    Z_F64_EMU_ANISO_FAR = 8,  // spacings more than 16 apart: one rounded product per axis
};

struct ZParams {
    int64_t nx, ny, nz;
    int64_t pitch;  // elements between consecutive rows (nx for a contiguous grid)
    int kchunk, ntx;
    EmuCoef ek;
    float fdtlam, fax, fay, faz;
};

// True when the TMA path can serve this grid and these pointers.
bool zmarch_supported(Grid3 g, int esz, const void *a, const void *b, const void *c);
// The same for one forward step, unless PS_OVERRIDE_STEP_PLAIN asks for the plain kernel.
bool step_tma_ok(Grid3 g, int esz, const void *a, const void *b, const void *c);
// The same for rows that are no multiple of 16 bytes, staged row by row (zrag_tile.cuh): any
// nx, fewer than 2^31 elements.
bool ragged_supported(Grid3 g, const void *a, const void *b, const void *c);
bool step_ragged_ok(Grid3 g, int esz, const void *a, const void *b, const void *c);
bool comp_ragged_ok(Grid3 g, const void *a, const void *b, const void *c);  // the two-float step
// Map over n consecutive elements: rows of rowlen (a multiple of 16 bytes; a last part of a
// row is left out) with a box of bx x by, or with by = 0 one line with a box of bx.
bool make_tensor_map_rows(CUtensorMap *m, const void *ptr, int esz, int64_t n, int64_t rowlen, unsigned bx,
                          unsigned by);
// Map over the FP32 grid's rows r, r+4, ... (flat rows y + ny*z, r < 4) with a box of bx x by; row r
// starts at element (r*nx + the field's first element in its 16 bytes) mod 4 of the map's rows.
bool make_tensor_map_quarter(CUtensorMap *m, const float *ptr, Grid3 g, int64_t r, unsigned bx, unsigned by);
// The four such maps (by flat row mod 4) of N fields.
template <int N>
struct RagMaps {
    CUtensorMap f[N][4];
};
// Planes per chunk of the FP32 pair kernels for `tiles` tiles on `slots` resident CTAs.
int pair_kchunk(Grid3 g, int64_t tiles, int64_t slots);
// Grids whose steps take the column kernels (stencil_basic.cuh), aligned ones inside a time loop only; mode:
// Z_F32, Z_F32_COMP, Z_F64_SCALED, Z_F64_EMU_ISO (Ci as given, equal spacings) or Z_F64_EMU_ANISO (any
// unequal spacings).
bool step_small(Grid3 g, int mode, bool in_loop);
// Useful lanes of the staged two-float step on odd rows against the column kernel's.
double comp_ragged_share(Grid3 g);
// Whether fused FP32 pairs (zpair.cu) beat single steps in a loop on this grid; states: a
// loop that keeps every state.
bool pairs_pay(Grid3 g, bool states);
bool pairs_pay_ragged(Grid3 g);  // on rows that are no multiple of 16 bytes
// 3-D tiled tensor map over a (nz, ny, nx) field with a bx x by x 1 box.
bool make_tensor_map_3d(CUtensorMap *m, const void *ptr, int esz, Grid3 g, unsigned bx, unsigned by);
// The same over a grid whose rows are `pitch` elements apart (pitch*esz a multiple of 16).
bool make_tensor_map_3d_pitch(CUtensorMap *m, const void *ptr, int esz, Grid3 g, int64_t pitch,
                              unsigned bx, unsigned by);
// True when the driver's tensor-map encoder could be loaded (a GPU driver is present).
bool tma_encoder_available();
// Whether the pre-scaled FP64 step takes the four-nodes-per-thread kernel (rows of a multiple
// of 32 bytes whose length suits its 128-node tiles, 32-byte aligned fields).
bool f64_scaled_wide(Grid3 g, const void *T2, const void *T, const void *Ci);
// Step parameters of the z-march kernels for coefficients c on grid g with row pitch `pitch`.
ZParams zparams_for(StepCoef c, Grid3 g, int64_t pitch);

// TMA-fed transposed step (adjoint_zmarch.cu).
bool adjoint_zmarch_supported(Grid3 g, int esz, const void *const *ptrs, int nptr);
template <typename E>
cudaError_t launch_adjoint_zmarch(E *Tbar, E *Cibar, const E *ybar, const E *T, const E *Ci,
                                  StepCoef c, Grid3 g, cudaStream_t s);
unsigned adjoint_device_error(bool clear);
// TMA-fed transposed step on the pre-scaled coefficient (adjoint_scaled.cu).
cudaError_t launch_adjoint_scaled(double *Tbar, double *Csbar, const double *ybar, const double *T,
                                  const double *Cs, Grid3 g, cudaStream_t s);
// The same kernel on Ci as given: equal spacings, or the axes' coefficients at one exponent
// (ek.axes other than AX_FAR).
cudaError_t launch_adjoint_given(double *Tbar, double *Cibar, const double *ybar, const double *T,
                                 const double *Ci, const EmuCoef &ek, Grid3 g, cudaStream_t s);
// True when dt*lam*_d^2 is positive and normal on every axis (the emulated FP64 forms).
bool emu_ok(StepCoef c);
// One step of the TMA z-march in `mode`; E2 / Ein: the correction fields of the
// two-float state (Z_F32_COMP only, else unused).  write_bnd: also store the x and y
// boundary nodes of planes 1 .. nz-2 as copies of T's (not with Z_F32_COMP).
cudaError_t launch_zmarch(int mode, void *T2, const void *T, void *E2, const void *Ein, const void *Ci,
                          StepCoef c, Grid3 g, cudaStream_t s, bool write_bnd = false);
// The same on ragged rows (mode: Z_F64_EMU_ISO, Z_F64_EMU_ANISO, Z_F64_SCALED or Z_F32;
// the caller has checked step_ragged_ok).
cudaError_t launch_zmarch_ragged(int mode, void *T2, const void *T, const void *Ci, StepCoef c, Grid3 g,
                                 cudaStream_t s, bool write_bnd = false);
unsigned zmarch_device_error(bool clear);
// One step of the two-float state on ragged rows (zcomp_rag.cu); the caller has checked comp_ragged_ok
// of T2, T and Ci.  E and E2 may start at any element.
cudaError_t launch_comp_ragged(float *T2, const float *T, float *E2, const float *E, const float *Ci, StepCoef c,
                               Grid3 g, cudaStream_t s);

}  // namespace psd

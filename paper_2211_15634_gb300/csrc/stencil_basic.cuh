// Plain 7-point step kernels: one thread per interior (i, j) column,
// marching along z with a three-value register queue.  x/y neighbours are
// read through the L1/L2 caches.
//
// They serve two kinds of grid.  Small ones (step_small, zmarch.cu; rows of a multiple of 16
// bytes inside a time loop only): a march of 1 .. 16 planes per thread keeps a step at a few
// memory round trips, where the TMA z-march waits for 8 planes of copies one after the other.
// Measured, us a step in a captured loop (march of 8 planes / this): FP64 pre-scaled 32^3 7.6 /
// 1.7, 64^3 7.6 / 3.2, 96^3 9.1 / 6.3, 128^3 14.9 / 10.5; FP32 32^3 4.2 / 1.5, 64^3 4.3 / 2.2,
// 96^3 4.4 / 3.6, 160^3 10.9 / 8.8, 192^3 14.3 / 13.7, 208^3 19 / 22.  And grids
// that the march cannot take or would be slower on (2^31 nodes and more on ragged rows, spacings
// more than 16 apart on odd nx, plain FP64; FP32 grids on ragged rows that leave many lanes of
// its tiles idle: step_ragged_ok, comp_ragged_ok).
// They never store boundary nodes: x faces stored beside the interior cost more than the
// boundary copy they save (127^3 FP32 states: 10.1 us a step against 8.3).
// The next step's CTAs are let in at the end of the march, not at its start: with one wave of
// CTAs or less they would fill whatever slots are free and leave the SMs unevenly loaded
// (FP32 160 x 63 x 311: 9.0 us against 7.5).
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#include "emu64.cuh"
#include "internal.h"
#include "node.cuh"
#include "pdl.cuh"
#include "waves.h"

namespace psd {

template <typename F>
struct CoefT {
    F dtlam, ax, ay, az;
};

// FP64 data with the one-DFMA emulated arithmetic of emu64.cuh.
template <int kAx, bool kScaled>
__global__ void __launch_bounds__(256)
k_step_basic_emu(double *__restrict__ T2, const double *__restrict__ T,
                 const double *__restrict__ Ci, EmuCoef c, int64_t nx, int64_t ny, int64_t nz,
                 int kchunk) {
    grid_dep_wait();  // the previous step's writes (and its reads of T2) are complete
    const int64_t i = 1 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t j = 1 + (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    if (i > nx - 2 || j > ny - 2) return;
    const int64_t k0 = 1 + (int64_t)blockIdx.z * kchunk;
    const int64_t k1 = k0 + kchunk < nz - 1 ? k0 + kchunk : nz - 1;
    if (k0 >= k1) return;
    const int64_t sy = nx, sz = nx * ny;
    const unsigned long long *__restrict__ Tb = (const unsigned long long *)T;
    int64_t p = i + sy * (j + ny * k0);
    unsigned long long tm = Tb[p - sz], tc = Tb[p];
    for (int64_t k = k0; k < k1; ++k, p += sz) {
        const unsigned long long tp = Tb[p + sz], xm = Tb[p - 1], xp = Tb[p + 1], ym = Tb[p - sy], yp = Tb[p + sy];
        if (kScaled)  // Ci holds dt*lam*_d^2*Ci (isotropic grid)
            T2[p] = emu_step_node_scaled(tc, xm, xp, ym, yp, tm, tp, Ci[p]);
        else
            T2[p] = emu_step_node<kAx, false>(tc, xm, xp, ym, yp, tm, tp, Ci[p], c);
        tm = tc;
        tc = tp;
    }
    grid_dep_launch();
}

// Fig. 1 step!: T2 = T + dt*lam*Ci*((d2x*_dx^2 + d2y*_dy^2) + d2z*_dz^2) at
// interior nodes; the z-range of this block is [k0, k1).  FP32: f32_node's roundings.
// kComp (FP32): the state is the two-float pair (T, E) and (T2, E2) receives the
// compensated step (comp32_node, node.cuh).
template <typename F, bool kComp>
__global__ void __launch_bounds__(256)
k_step_basic(F *__restrict__ T2, const F *__restrict__ T, F *__restrict__ E2,
             const F *__restrict__ E, const F *__restrict__ Ci, CoefT<F> c, int64_t nx, int64_t ny,
             int64_t nz, int kchunk) {
    grid_dep_wait();
    const int64_t i = 1 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t j = 1 + (int64_t)blockIdx.y * blockDim.y + threadIdx.y;
    if (i > nx - 2 || j > ny - 2) return;
    const int64_t k0 = 1 + (int64_t)blockIdx.z * kchunk;
    const int64_t k1 = k0 + kchunk < nz - 1 ? k0 + kchunk : nz - 1;
    if (k0 >= k1) return;
    const int64_t sy = nx, sz = nx * ny;
    int64_t p = i + sy * (j + ny * k0);
    F tm = T[p - sz], tc = T[p];
    for (int64_t k = k0; k < k1; ++k, p += sz) {
        const F tp = T[p + sz];
        if constexpr (kComp) {
            float e2;
            T2[p] = comp32_node(tc, T[p - 1], T[p + 1], T[p - sy], T[p + sy], tm, tp, E[p], E[p - 1],
                                E[p + 1], E[p - sy], E[p + sy], E[p - sz], E[p + sz], Ci[p], c.dtlam,
                                c.ax, c.ay, c.az, &e2);
            E2[p] = e2;
        } else {
            const F xm = T[p - 1], xp = T[p + 1], ym = T[p - sy], yp = T[p + sy];
            if constexpr (sizeof(F) == 4) {
                T2[p] = f32_node(tc, xm, xp, ym, yp, tm, tp, Ci[p], c.dtlam, c.ax, c.ay, c.az);
            } else {
                const F d2x = (xp - tc) - (tc - xm);
                const F d2y = (yp - tc) - (tc - ym);
                const F d2z = (tp - tc) - (tc - tm);
                const F lap = (d2x * c.ax + d2y * c.ay) + d2z * c.az;
                T2[p] = tc + c.dtlam * (Ci[p] * lap);
            }
        }
        tm = tc;
        tc = tp;
    }
    grid_dep_launch();
}

// Launch shape of the column kernels: 32 x 8 columns per CTA and kchunk planes.  false: the
// grid does not fit a launch.
enum ColumnKind { COL_F64, COL_F32, COL_COMP };
inline bool column_shape(int64_t nx, int64_t ny, int64_t nz, ColumnKind kind, bool small, dim3 *grid, int *kchunk) {
    const int64_t gx = (nx - 2 + 31) / 32, gy = (ny - 2 + 7) / 8;
    // about 8 blocks per SM, each chunk at least 16 planes
    const int64_t want = (8LL * sm_count() + gx * gy - 1) / (gx * gy);
    int64_t kc = (nz - 2 + want - 1) / want;
    if (kc < 16) kc = 16;
    if (small) {
        // FP64 and the two-float step: about eight CTAs per SM, 1 to 8 planes.  FP32: the
        // planes of a chunk are loaded four at a time (the compiler's unrolling), so 4, 8 or
        // the long chunks, and 1 where even that leaves SMs idle.  Sweeps at 32^3 .. 192^3:
        // within 10% of the best chunk at each.
        const int64_t planes = gx * gy * (nz - 2);  // CTAs at one plane each
        if (kind == COL_F32) {
            const double r = (double)planes / (2.0 * sm_count());
            if (r < 16.0) kc = r < 1.0 ? 1 : (r < 6.0 ? 4 : 8);
        } else {
            kc = planes / (8LL * sm_count());
            if (kind == COL_COMP && kc > 8) {
                // long chunks that just fit eight CTAs per SM: 145 x 200 x 160 18.3 us a step, 19.4 in 8
                // planes, 193 x 100 x 250 18.7 and 19.8, 190 x 100 x 150 12.0 and 12.8
                while (gx * gy * ((nz - 2 + kc - 1) / kc) > 8LL * sm_count() && kc < nz) ++kc;
            } else {
                kc = kc < 1 ? 1 : (kc > 8 ? 8 : kc);
            }
        }
    }
    kc = grid_chunk(nz, (int)kc);
    const int64_t gz = (nz - 2 + kc - 1) / kc;
    if (gx > 0x7fffffff || gy > 65535 || gz > 65535) return false;
    *grid = dim3((unsigned)gx, (unsigned)gy, (unsigned)gz);
    *kchunk = (int)kc;
    return true;
}

template <int kAx, bool kScaled>
inline cudaError_t launch_basic_emu_t(double *T2, const double *T, const double *Ci, const EmuCoef &c, Grid3 g,
                                      cudaStream_t s, bool small) {
    dim3 grid;
    int kc;
    if (!column_shape(g.nx, g.ny, g.nz, COL_F64, small, &grid, &kc)) return cudaErrorInvalidConfiguration;
    return launch_pdl(k_step_basic_emu<kAx, kScaled>, grid, dim3(32, 8), 0, s, T2, T, Ci, c, g.nx, g.ny, g.nz, kc);
}

inline cudaError_t launch_step_basic_emu(double *T2, const double *T, const double *Ci, const EmuCoef &c, bool iso,
                                         Grid3 g, cudaStream_t s, bool scaled, bool small) {
    if (scaled) return launch_basic_emu_t<AX_ISO, true>(T2, T, Ci, c, g, s, small);
    if (iso) return launch_basic_emu_t<AX_ISO, false>(T2, T, Ci, c, g, s, small);
    if (c.axes == AX_COMMON) return launch_basic_emu_t<AX_COMMON, false>(T2, T, Ci, c, g, s, small);
    if (c.axes == AX_SPREAD) return launch_basic_emu_t<AX_SPREAD, false>(T2, T, Ci, c, g, s, small);
    return launch_basic_emu_t<AX_FAR, false>(T2, T, Ci, c, g, s, small);
}

template <typename F, bool kComp>
cudaError_t launch_step_basic(F *T2, const F *T, F *E2, const F *E, const F *Ci, CoefT<F> c, Grid3 g,
                              cudaStream_t s, bool small) {
    dim3 grid;
    int kc;
    if (!column_shape(g.nx, g.ny, g.nz, sizeof(F) == 8 ? COL_F64 : kComp ? COL_COMP : COL_F32, small, &grid, &kc)) return cudaErrorInvalidConfiguration;
    return launch_pdl(k_step_basic<F, kComp>, grid, dim3(32, 8), 0, s, T2, T, E2, E, Ci, c, g.nx, g.ny, g.nz, kc);
}

}  // namespace psd

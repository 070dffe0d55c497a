// 2-D form of the step (Fig. 1's step! with the z term dropped) as a warp-level
// y-march.
//
// Warp w owns a strip of 32*PX columns (PX nodes per lane: two 16-byte accesses when
// the rows allow them - eight FP32 or four FP64 nodes - else PX nodes 32 apart) and a chunk of
// interior rows [j0, j1).  Each
// lane keeps its own values of rows j-1, j, j+1 and Ci of row j in registers and
// loads row j+2 and Ci of row j+1 while it computes row j: plain coalesced loads,
// no shared memory and no barriers - the x-neighbours come from the neighbouring
// lanes by warp shuffles and, at the strip's two edges, from one extra load each.
// Every T value is read from HBM once (the strip-edge columns and the rows shared
// by consecutive chunks hit in L2).  The per-node arithmetic is the 3-D step's
// (node.cuh, emu64.cuh) with the z-neighbours set to the centre value: the z
// difference is then exactly zero.
#include <algorithm>

#include "emu64.cuh"
#include "internal.h"
#include "node.cuh"
#include "pdl.cuh"
#include "zmarch.h"

namespace psd {

struct P2D {
    int64_t nx, ny;
    int chunk, nstrips;
    float fdtlam, fax, fay;
    EmuCoef ek;
};

template <int MODE>
struct M2D;  // element type per mode
template <>
struct M2D<Z_F32> {
    using E = float;
};
template <>
struct M2D<Z_F64_SCALED> {
    using E = double;
};
template <>
struct M2D<Z_F64_EMU_ISO_DMUL> {
    using E = double;
};
template <>
struct M2D<Z_F64_EMU_ANISO> {
    using E = double;
};
template <>
struct M2D<Z_F64_EMU_ANISO_SPREAD> : M2D<Z_F64_EMU_ANISO> {};
template <>
struct M2D<Z_F64_NATIVE> {
    using E = double;
};

template <int MODE, typename E>
__device__ __forceinline__ E node2d(E c, E xm, E xp, E ym, E yp, E ci, const P2D &p) {
    if constexpr (MODE == Z_F32) {
        return f32_node(c, xm, xp, ym, yp, c, c, ci, p.fdtlam, p.fax, p.fay, 0.f);
    } else if constexpr (MODE == Z_F64_SCALED) {
        return f64s_node(c, xm, xp, ym, yp, c, c, ci);
    } else if constexpr (MODE == Z_F64_EMU_ISO_DMUL) {
        return emu_step_node<AX_ISO, true>(dbits(c), dbits(xm), dbits(xp), dbits(ym), dbits(yp), dbits(c),
                                           dbits(c), ci, p.ek);
    } else if constexpr (MODE == Z_F64_EMU_ANISO || MODE == Z_F64_EMU_ANISO_SPREAD) {
        constexpr int kAx = MODE == Z_F64_EMU_ANISO ? AX_COMMON : AX_SPREAD;
        return emu_step_node<kAx, false, 2>(dbits(c), dbits(xm), dbits(xp), dbits(ym), dbits(yp), dbits(c),
                                            dbits(c), ci, p.ek);
    } else {
        const double d2x = (xp - c) - (c - xm), d2y = (yp - c) - (c - ym);
        return c + p.ek.dtlam * (ci * (d2x * p.ek.ax + d2y * p.ek.ay));
    }
}

// PX values of row r starting at column x (x % PX == 0); columns >= nx read as 0
template <typename E, int PX>
__device__ __forceinline__ void load_row(E (&v)[PX], const E *__restrict__ A, int64_t r, int64_t nx,
                                         int64_t x) {
    const E *q = A + r * nx + x;
    if constexpr (PX * sizeof(E) == 32) {  // two 16-byte loads
        if (x + PX <= nx) {
            if constexpr (sizeof(E) == 8) {
                const double2 a = __ldg((const double2 *)q), b = __ldg((const double2 *)q + 1);
                v[0] = a.x;
                v[1] = a.y;
                v[2] = b.x;
                v[3] = b.y;
            } else {
                const float4 a = __ldg((const float4 *)q), b = __ldg((const float4 *)q + 1);
                v[0] = a.x;
                v[1] = a.y;
                v[2] = a.z;
                v[3] = a.w;
                v[4] = b.x;
                v[5] = b.y;
                v[6] = b.z;
                v[7] = b.w;
            }
            return;
        }
    }
    if constexpr (PX * sizeof(E) == 16) {
        if (x + PX <= nx) {
            if constexpr (sizeof(E) == 8) {
                const double2 t = __ldg((const double2 *)q);
                v[0] = t.x;
                v[1] = t.y;
            } else {
                const float4 t = __ldg((const float4 *)q);
                v[0] = t.x;
                v[1] = t.y;
                v[2] = t.z;
                v[3] = t.w;
            }
            return;
        }
    }
#pragma unroll
    for (int i = 0; i < PX; ++i) v[i] = x + i < nx ? __ldg(q + i) : E(0);
}

// The same for a lane's strided nodes x, x + 32, ..
template <typename E, int PX>
__device__ __forceinline__ void load_strided(E (&v)[PX], const E *__restrict__ A, int64_t r, int64_t nx, int64_t x) {
    const E *q = A + r * nx + x;
#pragma unroll
    for (int i = 0; i < PX; ++i) v[i] = x + 32 * i < nx ? __ldg(q + 32 * i) : E(0);
}

// MINB CTAs of 8 warps per SM: 3 for two FP64 / eight FP32 nodes per lane and the
// scalar forms (the FP64 emulated modes spill at 4, measured 4% slower there); 2 for four
// FP64 nodes per lane (111 registers, no spill)
// XS: distance between a lane's nodes - 1, neighbours (16-byte accesses), or 32, for rows at
// any element: consecutive lanes on consecutive elements, so that scalar accesses still fill
// whole sectors, and the loop's own instructions count for PX nodes.
template <int MODE, int PX, int MINB, int XS>
__global__ void __launch_bounds__(256, MINB)
k_ymarch2d(typename M2D<MODE>::E *__restrict__ T2, const typename M2D<MODE>::E *__restrict__ T,
           const typename M2D<MODE>::E *__restrict__ Ci, const P2D p) {
    using E = typename M2D<MODE>::E;
    grid_dep_wait();  // the previous step's writes (and its reads of T2) are complete
    const int lane = threadIdx.x & 31;
    const int64_t warp = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t strip = warp % p.nstrips, chunk = warp / p.nstrips;
    const int64_t nx = p.nx, ny = p.ny;
    const int64_t j0 = 1 + chunk * p.chunk, j1 = min(j0 + p.chunk, ny - 1);  // rows [j0, j1)
    if (j0 >= j1) return;  // warp-uniform
    const int64_t x0 = strip * 32 * PX, gx0 = x0 + lane * (XS == 1 ? PX : 1);
    const bool has_l = lane == 0 && x0 >= 1, has_r = lane == 31 && x0 + 32 * PX < nx;
    bool wr[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) wr[i] = gx0 + XS * i >= 1 && gx0 + XS * i <= nx - 2;
    const bool all_w = gx0 >= 1 && gx0 + XS * (PX - 1) <= nx - 2;
    auto load = [&](E (&v)[PX], const E *__restrict__ A, int64_t r) {
        if constexpr (XS == 1)
            load_row<E, PX>(v, A, r, nx, gx0);
        else
            load_strided<E, PX>(v, A, r, nx, gx0);
    };

    E up[PX], c[PX], dn[PX], ci[PX], nxt[PX], cin[PX];
    load(up, T, j0 - 1);
    load(c, T, j0);
    load(dn, T, j0 + 1);
    load(ci, Ci, j0);
    E hl = has_l ? __ldg(T + j0 * nx + x0 - 1) : E(0), hr = has_r ? __ldg(T + j0 * nx + x0 + 32 * PX) : E(0);
    for (int64_t j = j0; j < j1; ++j) {
        // row j+2 (the next "down" row) and Ci of row j+1, and the strip-edge values of
        // row j+1, are in flight while row j is computed
        const bool more = j + 1 < j1;
        if (more) {
            load(nxt, T, j + 2);
            load(cin, Ci, j + 1);
        }
        const E hl1 = (more && has_l) ? __ldg(T + (j + 1) * nx + x0 - 1) : E(0);
        const E hr1 = (more && has_r) ? __ldg(T + (j + 1) * nx + x0 + 32 * PX) : E(0);
        // x-neighbours: a lane's own or the neighbouring lanes' (strided: the neighbouring lane's
        // node of the same group of 32, at its ends of the group beside it)
        E xl[PX], xr[PX];
        if constexpr (XS == 1) {
            xl[0] = __shfl_up_sync(0xffffffffu, c[PX - 1], 1);
            xr[PX - 1] = __shfl_down_sync(0xffffffffu, c[0], 1);
            if (lane == 0) xl[0] = hl;
            if (lane == 31) xr[PX - 1] = hr;
#pragma unroll
            for (int i = 1; i < PX; ++i) {
                xl[i] = c[i - 1];
                xr[i - 1] = c[i];
            }
        } else {
            E pl = hl, pr = hr;
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                const E v = __shfl_sync(0xffffffffu, c[i], (lane + 31) & 31);
                xl[i] = lane == 0 ? pl : v;
                pl = v;
            }
#pragma unroll
            for (int i = PX - 1; i >= 0; --i) {
                const E v = __shfl_sync(0xffffffffu, c[i], (lane + 1) & 31);
                xr[i] = lane == 31 ? pr : v;
                pr = v;
            }
        }
        E out[PX];
        bool warp_fast = false;
        if constexpr (MODE == Z_F64_SCALED || MODE == Z_F64_EMU_ISO_DMUL || MODE == Z_F64_EMU_ANISO ||
                      MODE == Z_F64_EMU_ANISO_SPREAD) {
            // one same-binade check over this lane's distinct values (words of nodes that
            // are not written replaced by the reference, so they cannot force the general
            // path); the whole warp takes the short path together when all lanes pass
            bool any_wr = false;
#pragma unroll
            for (int i = 0; i < PX; ++i) any_wr = any_wr || wr[i];
            // a lane that writes none of its nodes (past the grid) votes for the fast path:
            // its reference is 1.0's word (its outputs are never stored)
            // (strided lanes: the first node they write; node i's centre is no neighbour of theirs)
            unsigned hc = any_wr ? (unsigned)(dbits(c[0]) >> 32) : 0x3ff00000u;
            if constexpr (XS != 1 && PX > 1)
                if (any_wr && !wr[0]) hc = (unsigned)(dbits(c[1]) >> 32);
            unsigned hw[XS == 1 ? 3 * PX + 1 : 5 * PX];
            hw[0] = wr[0] ? (unsigned)(dbits(xl[0]) >> 32) : hc;
            hw[1] = wr[PX - 1] ? (unsigned)(dbits(xr[PX - 1]) >> 32) : hc;
#pragma unroll
            for (int i = 0; i < PX; ++i) {
                hw[2 + 2 * i] = wr[i] ? (unsigned)(dbits(up[i]) >> 32) : hc;
                hw[3 + 2 * i] = wr[i] ? (unsigned)(dbits(dn[i]) >> 32) : hc;
            }
#pragma unroll
            for (int i = 1; i < PX; ++i) {
                const bool need = wr[i] || (XS == 1 && (wr[i - 1] || (i + 1 < PX && wr[i + 1])));
                hw[1 + 2 * PX + i] = need ? (unsigned)(dbits(c[i]) >> 32) : hc;
            }
            if constexpr (XS != 1) {  // hw[3*PX + 1 ..]: the x-neighbours not among the words yet
#pragma unroll
                for (int i = 1; i < PX; ++i) {
                    hw[3 * PX + i] = wr[i] ? (unsigned)(dbits(xl[i]) >> 32) : hc;
                    hw[4 * PX + i - 1] = wr[i - 1] ? (unsigned)(dbits(xr[i - 1]) >> 32) : hc;
                }
                hw[5 * PX - 1] = hc;
            }
            warp_fast = __all_sync(0xffffffffu, emu_same_binade_hi(hw, hc));
        }
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            const E xm = xl[i], xp = xr[i];
            if constexpr (MODE == Z_F64_SCALED) {
                if (warp_fast) {
                    out[i] = emu_fast_node_scaled(dbits(c[i]), dbits(xm), dbits(xp), dbits(up[i]), dbits(dn[i]),
                                                  dbits(c[i]), dbits(c[i]), ci[i]);
                    continue;
                }
            } else if constexpr (MODE == Z_F64_EMU_ISO_DMUL) {
                if (warp_fast) {
                    out[i] = emu_fast_node<AX_ISO, true>(dbits(c[i]), dbits(xm), dbits(xp), dbits(up[i]),
                                                         dbits(dn[i]), dbits(c[i]), dbits(c[i]), ci[i], p.ek);
                    continue;
                }
            } else if constexpr (MODE == Z_F64_EMU_ANISO || MODE == Z_F64_EMU_ANISO_SPREAD) {
                if (warp_fast) {
                    constexpr int kAx = MODE == Z_F64_EMU_ANISO ? AX_COMMON : AX_SPREAD;
                    out[i] = emu_fast_node<kAx, false, 2>(dbits(c[i]), dbits(xm), dbits(xp), dbits(up[i]),
                                                          dbits(dn[i]), dbits(c[i]), dbits(c[i]), ci[i], p.ek);
                    continue;
                }
            }
            out[i] = node2d<MODE, E>(c[i], xm, xp, up[i], dn[i], ci[i], p);
        }
        E *q = T2 + j * nx + gx0;
        if constexpr (XS == 1 && PX * sizeof(E) == 32) {
            if (all_w) {
                if constexpr (sizeof(E) == 8) {
                    ((double2 *)q)[0] = make_double2(out[0], out[1]);
                    ((double2 *)q)[1] = make_double2(out[2], out[3]);
                } else {
                    ((float4 *)q)[0] = make_float4(out[0], out[1], out[2], out[3]);
                    ((float4 *)q)[1] = make_float4(out[4], out[5], out[6], out[7]);
                }
            } else {
#pragma unroll
                for (int i = 0; i < PX; ++i)
                    if (wr[i]) q[i] = out[i];
            }
        } else if constexpr (XS == 1 && PX * sizeof(E) == 16) {
            if (all_w) {
                if constexpr (sizeof(E) == 8)
                    *(double2 *)q = make_double2(out[0], out[1]);
                else
                    *(float4 *)q = make_float4(out[0], out[1], out[2], out[3]);
            } else {
#pragma unroll
                for (int i = 0; i < PX; ++i)
                    if (wr[i]) q[i] = out[i];
            }
        } else {
#pragma unroll
            for (int i = 0; i < PX; ++i)
                if (wr[i]) q[XS * i] = out[i];
        }
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            up[i] = c[i];
            c[i] = dn[i];
            dn[i] = nxt[i];
            ci[i] = cin[i];
        }
        hl = hl1;
        hr = hr1;
    }
    grid_dep_launch();  // at the end: less than a wave of CTAs would else fill up unevenly
}

// Edges of a 2-D field: T2 = T on rows 0, ny-1 and columns 0, nx-1 (Fig. 1's
// T2 = copy(T) as far as the boundary is concerned).
template <typename E>
__global__ void k_copy_edges2d(E *__restrict__ T2, const E *__restrict__ T, int64_t nx, int64_t ny) {
    const int64_t n_edge = 2 * nx + 2 * (ny - 2);
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n_edge;
         t += (int64_t)gridDim.x * blockDim.x) {
        int64_t p;
        if (t < nx) p = t;
        else if (t < 2 * nx) p = (ny - 1) * nx + (t - nx);
        else {
            const int64_t u = t - 2 * nx, r = 1 + u / 2;
            p = r * nx + ((u & 1) ? nx - 1 : 0);
        }
        T2[p] = T[p];
    }
}

template <int MODE, int PX, int MINB = 3, int XS = 1>
static cudaError_t launch_2d_t(void *T2, const void *T, const void *Ci, P2D p, int64_t nx, int64_t ny,
                               cudaStream_t s) {
    using E = typename M2D<MODE>::E;
    p.nx = nx;
    p.ny = ny;
    p.nstrips = (int)((nx + 32 * PX - 1) / (32 * PX));
    int chunk = launch_override(PS_OVERRIDE_CHUNK2D);
    if (chunk <= 0) {
        // A row's loads come one row ahead, so a chunk is a chain of round trips: on small grids
        // one or two rows per warp, a few where the warps make some waves, and about eight
        // waves of long chunks (which re-read two rows each) only on large ones.  us a step
        // against the 16 rows small grids had: FP64 512^2 3.1 / 14, 1024^2 6.5 / 14, 2048^2
        // 19.8 / 20.2; FP32 512^2 2.2 / 8.4, 1024^2 3.3 / 8.3, 4096^2 34 / 39.
        const int64_t rows = (ny - 2) * (int64_t)p.nstrips;  // warps at one row each
        const double waves = (double)rows / (8.0 * MINB * sm_count());
        const int64_t c = rows / (8LL * 48 * sm_count());
        chunk = waves <= 1.0 ? 1 : (waves <= 2.0 ? 2 : (waves <= 32.0 ? 4 : (int)(c < 8 ? 8 : (c > 256 ? 256 : c))));
    }
    p.chunk = chunk;
    const int64_t nch = (ny - 2 + chunk - 1) / chunk, warps = nch * p.nstrips, blocks = (warps + 7) / 8;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    return launch_pdl(k_ymarch2d<MODE, PX, MINB, XS>, dim3((unsigned)blocks), dim3(256), 0, s, (E *)T2, (const E *)T,
                      (const E *)Ci, p);
}

template <int MODE>
static cudaError_t launch_aniso2d(bool vec, void *T2, const void *T, const void *Ci, P2D p, int64_t nx, int64_t ny,
                                  cudaStream_t s) {
    if (!vec) return launch_2d_t<MODE, 2, 4, 32>(T2, T, Ci, p, nx, ny, s);
    // bound by issue, so more warps with fewer nodes each once there are many rows:
    // 6000 x 8192 245 us, 255 with four per lane; 2048^2 29 and 28
    if (nx * ny >= (1LL << 24)) return launch_2d_t<MODE, 2, 4>(T2, T, Ci, p, nx, ny, s);
    return launch_2d_t<MODE, 4, 2>(T2, T, Ci, p, nx, ny, s);
}

// mode: Z_F32, Z_F64_SCALED (Ci holds dt*lam*_dx^2*Ci, equal spacings), Z_F64_EMU_ISO_DMUL
// (equal spacings, positive coefficient), Z_F64_EMU_ANISO (unequal ones within a factor of
// 16) or Z_F64_NATIVE (anything else in FP64)
cudaError_t launch_step2d(int mode, void *T2, const void *T, const void *Ci, StepCoef c, int64_t nx,
                          int64_t ny, cudaStream_t s) {
    P2D p{};
    p.fdtlam = (float)c.dtlam;
    p.fax = (float)c.ax;
    p.fay = (float)c.ay;
    p.ek = emu_coef(c.dtlam, c.ax, c.ay, c.ax);  // the z term is not used
    p.ek.az = 0.0;                               // (and vanishes in the general path's plain form)
    const int esz = mode == Z_F32 ? 4 : 8;
    const bool vec = ((nx * esz) % 16 == 0) && ((((uintptr_t)T2 | (uintptr_t)T | (uintptr_t)Ci) & 15u) == 0);
    // Rows at any element take strided lanes (us a step at 6000 x 8191 against one node per lane:
    // FP64 pre-scaled 265 / 323, unequal spacings 313 / 359, FP32 106 / 227).
    switch (mode) {
        case Z_F32:
            // eight nodes per lane (two 16-byte accesses): measured 7-9% faster than four at
            // 16384^2 and 32768^2; strided four at four CTAs per SM (eight at three spill: 128 us)
            return vec ? launch_2d_t<Z_F32, 8>(T2, T, Ci, p, nx, ny, s)
                       : launch_2d_t<Z_F32, 4, 4, 32>(T2, T, Ci, p, nx, ny, s);
        // FP64: four nodes per lane (two 16-byte accesses) at two CTAs per SM, measured 8%
        // faster than two per lane at three CTAs per SM at 16384^2 (6% at 8192^2); four per
        // lane at three CTAs per SM spilled and ran 25% slower.  Strided: two at four CTAs (four
        // at two: 273 us)
        case Z_F64_SCALED:
            return vec ? launch_2d_t<Z_F64_SCALED, 4, 2>(T2, T, Ci, p, nx, ny, s)
                       : launch_2d_t<Z_F64_SCALED, 2, 4, 32>(T2, T, Ci, p, nx, ny, s);
        case Z_F64_EMU_ISO_DMUL:
            return vec ? launch_2d_t<Z_F64_EMU_ISO_DMUL, 4, 2>(T2, T, Ci, p, nx, ny, s)
                       : launch_2d_t<Z_F64_EMU_ISO_DMUL, 2, 4, 32>(T2, T, Ci, p, nx, ny, s);
        // spacings within a factor of 16 of each other; beyond that plain FP64, whose products
        // lose nothing at any ratio
        case Z_F64_EMU_ANISO:
            if (p.ek.axes == AX_COMMON) return launch_aniso2d<Z_F64_EMU_ANISO>(vec, T2, T, Ci, p, nx, ny, s);
            if (p.ek.axes == AX_SPREAD) return launch_aniso2d<Z_F64_EMU_ANISO_SPREAD>(vec, T2, T, Ci, p, nx, ny, s);
            break;
        default:
            break;
    }
    return vec ? launch_2d_t<Z_F64_NATIVE, 4, 2>(T2, T, Ci, p, nx, ny, s)
               : launch_2d_t<Z_F64_NATIVE, 1>(T2, T, Ci, p, nx, ny, s);
}

cudaError_t launch_copy_edges2d(void *T2, const void *T, int64_t nx, int64_t ny, int esz, cudaStream_t s) {
    const int64_t n = 2 * nx + 2 * (ny - 2);
    const unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, 4096);
    if (esz == 8)
        k_copy_edges2d<unsigned long long><<<blocks, 256, 0, s>>>((unsigned long long *)T2,
                                                                 (const unsigned long long *)T, nx, ny);
    else
        k_copy_edges2d<unsigned><<<blocks, 256, 0, s>>>((unsigned *)T2, (const unsigned *)T, nx, ny);
    return cudaGetLastError();
}

}  // namespace psd

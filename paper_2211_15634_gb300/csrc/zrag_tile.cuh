// Body of the z-march step on ragged rows: grids whose row length is not a multiple of
// 16 bytes, so that no 2-D or 3-D tensor map can describe them (odd nx in FP64, nx % 4 != 0
// in FP32).
//
// The march, the ring of NST plane stages and the per-node arithmetic are zmarch_tile.cuh's;
// what differs is how a plane gets into its stage.
//  * FP64 (odd nx): two rows together are a multiple of 16 bytes, so the field is mapped as
//    rows of 2*nx, and a plane of the tile arrives as two boxes of T and two of Ci: its even
//    and its odd tile rows.  (A last single row is outside the map and reads as zeros: it is
//    an edge of the last plane, which no interior node's stencil touches.)
//  * FP32: the field is mapped as one line of n elements and every row arrives as a copy of
//    its own, issued by the warp that owns the row (a copy's operands are uniform registers:
//    one warp issuing all 18 kept the others waiting at the barrier, 299 against 241 us at
//    511^3).  In FP64, bound by instruction issue, the copies' own instructions cost more
//    (255^3: 90 us, the column kernel's time).
// Every copy starts at the 16-byte boundary at or below its first element, so a row's data
// begins 0 .. P-1 elements (P = 16 bytes) into its slot, by (row * nx + X0 - 1) mod P, which
// every warp follows for its own row, the rows above and below and the next plane.
// Tiles start at the first interior node, not at the boundary: no box alignment binds them.
// Lanes own nodes lane + 32*i of their row rather than PX neighbours: with rows at any
// element there are no aligned vectors, and consecutive lanes on consecutive elements read
// shared memory without bank conflicts and store whole sectors.  Each x-neighbour is one
// more shared-memory read.
#pragma once

#include <cuda.h>

#include "emu64.cuh"
#include "node.cuh"
#include "tma.cuh"
#include "zmarch.h"
#include "zmarch_tile.cuh"

namespace psd {

// Sizes of a ragged tile of BY rows, PX nodes per lane; tile row h of T is at row(h), Ci's at
// crow(h), in elements from the stage's start.
template <int MODE, int PX, int BY>
struct ZRag {
    using E = typename ZTraits<MODE>::E;
    static constexpr bool kPairs = sizeof(E) == 8;               // row pairs, else single rows
    static constexpr int BX = 32 * PX, P = 16 / (int)sizeof(E), H = BY + 2;
    static constexpr int W = (BX + 2 + P - 1 + P - 1) / P * P;  // elements copied per row
    static constexpr unsigned RB = W * sizeof(E);                // bytes copied per row
    // a copy lands on 128 bytes: a box of H/2 (BY/2) rows, or a row
    static constexpr unsigned TBOX = ((kPairs ? H / 2 : 1) * RB + 127) / 128 * 128;
    static constexpr unsigned CBOX = ((kPairs ? BY / 2 : 1) * RB + 127) / 128 * 128;
    static constexpr unsigned CI0 = (kPairs ? 2 : H) * TBOX;     // Ci rows after T's
    static constexpr unsigned SB = CI0 + (kPairs ? 2 : BY) * CBOX;
    static_assert(!kPairs || BY % 2 == 0, "even and odd rows in equal boxes");
    static __device__ __forceinline__ int row(int h) {
        return kPairs ? (h & 1) * (int)(TBOX / sizeof(E)) + (h >> 1) * W : h * (int)(TBOX / sizeof(E));
    }
    static __device__ __forceinline__ int crow(int h) {
        return (int)(CI0 / sizeof(E)) + (kPairs ? (h & 1) * (int)(CBOX / sizeof(E)) + (h >> 1) * W
                                                : h * (int)(CBOX / sizeof(E)));
    }
};

// One CTA (32 * BY threads): output planes [k0, k1) of the BX x BY tile at (X0, Y0) (interior
// coordinates: the tile's first node is an interior one).  tmT / tmC: maps of T and Ci, rows
// of 2*nx with boxes of W x H/2 and W x BY/2 (FP64) or one line with a box of W (FP32).  kBnd: also the x and y boundary nodes of those planes, as T's.
template <int MODE, int PX, int BY, int NST, bool kBnd>
__device__ __forceinline__ void zrag_tile(const CUtensorMap *tmT, const CUtensorMap *tmC,
                                          void *__restrict__ T2v, const ZParams &p, int X0, int Y0, int k0,
                                          int k1, unsigned *err) {
    using R = ZRag<MODE, PX, BY>;
    using E = typename R::E;
    constexpr bool kF64 = sizeof(E) == 8;
    constexpr int H = R::H, P = R::P;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *bar = (uint64_t *)(smem + NST * R::SB);
    __shared__ int s_abort;
    const int lane = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int nx = (int)p.nx, ny = (int)p.ny;

    if (threadIdx.x == 0) {
        s_abort = 0;
        for (int s = 0; s < NST; ++s) mbar_init(&bar[s], R::kPairs ? 1 : BY);  // arrivals of the issuing threads
        fence_mbar_init();
    }
    __syncthreads();
    const int nplane = nx * ny;  // FP64: may wrap, used modulo P only
    // this thread's copies of plane q (q = k0-1 .. k1, stage (q - (k0-1)) % NST)
    auto issue = [&](int s, int q) {
        const bool ci = q >= k0 && q < k1;
        unsigned char *st = smem + s * R::SB;
        if constexpr (R::kPairs) {
            if (threadIdx.x != 0) return;
            mbar_expect_tx(&bar[s], R::RB * (H + (ci ? BY : 0)));
            // tile row h is field row r + h: the rows of one parity are consecutive pairs
            const int64_t r = (int64_t)q * ny + Y0 - 1;
            const int o = (int)(r & 1), g0 = (int)(r >> 1), g1 = (int)((r + 1) >> 1);
            const int x0 = (o * nx + X0 - 1) & ~1, x1 = ((o ^ 1) * nx + X0 - 1) & ~1;
            tma_load_2d(st, tmT, &bar[s], x0, g0);
            tma_load_2d(st + R::TBOX, tmT, &bar[s], x1, g1);
            if (ci) {  // Ci has no halo rows: its even rows are field rows r+1, r+3, ..
                tma_load_2d(st + R::CI0, tmC, &bar[s], x1, g1);
                tma_load_2d(st + R::CI0 + R::CBOX, tmC, &bar[s], x0, g0 + 1);
            }
        } else {  // the warp's own rows of T and Ci, the first and last warp also a halo row
            if (lane != 0) return;
            const bool edge = ty == 0 || ty == BY - 1;
            const int hrow = ty == 0 ? 0 : H - 1;
            mbar_expect_tx(&bar[s], R::RB * ((edge ? 2u : 1u) + (ci ? 1u : 0u)));
            const int e0 = q * nplane + (Y0 - 1) * nx + X0 - 1;  // tile row 0, column -1
            const int xo = (e0 + (ty + 1) * nx) & ~(P - 1);
            tma_load_1d(st + (ty + 1) * R::TBOX, tmT, &bar[s], xo);
            if (ci) tma_load_1d(st + R::CI0 + ty * R::CBOX, tmC, &bar[s], xo);
            if (edge) tma_load_1d(st + hrow * R::TBOX, tmT, &bar[s], (e0 + hrow * nx) & ~(P - 1));
        }
    };
    for (int s = 0; s < NST; ++s)
        if (k0 - 1 + s <= k1) issue(s, k0 - 1 + s);
    unsigned tpar = 0u;  // bit s: parity of the next completion of stage s
    auto tnext = [](int s) { return s + 1 == NST ? 0 : s + 1; };
    auto acquire = [&](int s) -> bool {
        const unsigned ph = (tpar >> s) & 1u;
        tpar ^= 1u << s;
        return mbar_wait(&bar[s], ph);
    };
    // After a timed-out wait: bounded waits for the copies of the last NST planes issued
    // (up to plane q_iss), so that no TMA write lands after the CTA exits.
    auto drain = [&](int q_iss) {
        for (int q = max(k0 - 1, q_iss - NST + 1); q <= q_iss; ++q) {
            const int i = q - (k0 - 1);
            mbar_wait(&bar[i % NST], (unsigned)(i / NST) & 1u);
        }
    };
    auto stage = [&](int s) { return (const E *)(smem + s * R::SB); };

    const int gy = Y0 + ty;
    // offset of a row's first element (tile column -1) in its slot, for the own row of plane k;
    // a row up or down and a plane on add -+nx and nx*ny
    int dk = ((k0 - 1) * nplane + gy * nx + X0 - 1) & (P - 1);
    const int dplane = nplane & (P - 1), drow = nx & (P - 1);
    auto at = [&](int s, int h, int d) { return stage(s) + R::row(h) + d + 1 + lane; };
    auto own = [&](int s, int d) { return at(s, ty + 1, d); };

    bool ok = acquire(0);
    E qm[PX], qc[PX];
#pragma unroll
    for (int i = 0; i < PX; ++i) qm[i] = own(0, dk)[32 * i];
    dk = (dk + dplane) & (P - 1);
    ok = acquire(1 % NST) && ok;
#pragma unroll
    for (int i = 0; i < PX; ++i) qc[i] = own(1 % NST, dk)[32 * i];
    if (!ok) {
        s_abort = 1;
        atomicOr(err, 1u);
    }
    __syncthreads();
    if (s_abort) {
        drain(min(k0 - 2 + NST, k1));
        return;
    }
    if (k0 - 1 + NST <= k1) issue(0, k0 - 1 + NST);  // stage 0 held plane k0-1

    const int gx0 = X0 + lane;
    const bool row_ok = gy <= ny - 2;
    bool use[PX], all_use = true;  // nodes this lane stores (32 apart)
#pragma unroll
    for (int i = 0; i < PX; ++i) {
        use[i] = gx0 + 32 * i <= nx - 2;
        all_use = all_use && use[i];
    }
    E *__restrict__ T2 = (E *)T2v;
    int sk = 1 % NST;  // stage of plane k
    int64_t base = (int64_t)gx0 + (int64_t)nx * ((int64_t)gy + (int64_t)ny * k0);

    const int64_t plane = (int64_t)nx * ny;

    for (int k = k0; k < k1; ++k, base += plane) {
        const int sk1 = tnext(sk), dk1 = (dk + dplane) & (P - 1);
        ok = acquire(sk1);  // plane k+1 (plane k, with its Ci, was acquired before)
        E qn[PX];
#pragma unroll
        for (int i = 0; i < PX; ++i) qn[i] = own(sk1, dk1)[32 * i];
        if (row_ok) {
            const E *Tc = own(sk, dk);
            const E *Tu = at(sk, ty, (dk - drow) & (P - 1)), *Td = at(sk, ty + 2, (dk + drow) & (P - 1));
            const E *Cc = stage(sk) + R::crow(ty) + dk + 1 + lane;
            E out[PX];
            if constexpr (kF64) {
                constexpr int kAx = MODE == Z_F64_EMU_ANISO ? AX_COMMON
                                    : MODE == Z_F64_EMU_ANISO_SPREAD ? AX_SPREAD : AX_ISO;
                constexpr bool kScaled = MODE == Z_F64_SCALED;
                unsigned long long c[PX], xm[PX], xp[PX], ym[PX], yp[PX], zm[PX], zp[PX];
                double ci[PX];
                unsigned hw[7 * PX - 1];
#pragma unroll
                for (int i = 0; i < PX; ++i) {
                    c[i] = dbits(qc[i]);
                    xm[i] = dbits(Tc[32 * i - 1]);
                    xp[i] = dbits(Tc[32 * i + 1]);
                    ym[i] = dbits(Tu[32 * i]);
                    yp[i] = dbits(Td[32 * i]);
                    zm[i] = dbits(qm[i]);
                    zp[i] = dbits(qn[i]);
                    ci[i] = Cc[32 * i];
                    hw[6 * i + 0] = (unsigned)(xm[i] >> 32);
                    hw[6 * i + 1] = (unsigned)(xp[i] >> 32);
                    hw[6 * i + 2] = (unsigned)(ym[i] >> 32);
                    hw[6 * i + 3] = (unsigned)(yp[i] >> 32);
                    hw[6 * i + 4] = (unsigned)(zm[i] >> 32);
                    hw[6 * i + 5] = (unsigned)(zp[i] >> 32);
                    if (i > 0) hw[6 * PX + i - 1] = (unsigned)(c[i] >> 32);
                }
                // a node that is not stored votes with the lane's first node's word, a lane
                // that stores none with 1.0's (see zmarch_tile.cuh); its nodes are the lane's last
                unsigned hc = (unsigned)(c[0] >> 32);
                if (!all_use) {
                    if (!use[0]) hc = 0x3ff00000u;
#pragma unroll
                    for (int i = 0; i < PX; ++i) {
                        if (use[i]) continue;
#pragma unroll
                        for (int j = 0; j < 6; ++j) hw[6 * i + j] = hc;
                        if (i > 0) hw[6 * PX + i - 1] = hc;
                    }
                }
                // warp-uniform paths, as in zmarch_tile.cuh
                if (__all_sync(0xffffffffu, emu_same_binade_hi(hw, hc))) {
#pragma unroll
                    for (int i = 0; i < PX; ++i) {
                        if constexpr (kScaled)
                            out[i] = emu_fast_node_scaled(c[i], xm[i], xp[i], ym[i], yp[i], zm[i], zp[i], ci[i]);
                        else
                            out[i] = emu_fast_node<kAx, false>(c[i], xm[i], xp[i], ym[i], yp[i], zm[i], zp[i],
                                                               ci[i], p.ek);
                    }
                } else {
                    unsigned ewin;
                    const bool near = __all_sync(0xffffffffu, emu_window_hi(hw, hc, &ewin));
#pragma unroll
                    for (int i = 0; i < PX; ++i) {
                        const unsigned long long c1[1] = {c[i]}, u1[1] = {ym[i]}, d1[1] = {yp[i]}, m1[1] = {zm[i]},
                                                 p1[1] = {zp[i]};
                        const double ci1[1] = {ci[i]};
                        double o[1];
                        if (near)
                            emu_lane_window<1, kScaled, kAx>(c1, xm[i], xp[i], u1, d1, m1, p1, ci1, p.ek, ewin, o);
                        else
                            emu_lane_general<1, kScaled, kAx>(c1, xm[i], xp[i], u1, d1, m1, p1, ci1, p.ek, o);
                        out[i] = o[0];
                    }
                }
            } else {
#pragma unroll
                for (int i = 0; i < PX; ++i)
                    out[i] = f32_node(qc[i], Tc[32 * i - 1], Tc[32 * i + 1], Tu[32 * i], Td[32 * i], qm[i], qn[i],
                                      Cc[32 * i], p.fdtlam, p.fax, p.fay, p.faz);
            }
#pragma unroll
            for (int i = 0; i < PX; ++i)
                if (use[i]) T2[base + 32 * i] = out[i];
            if constexpr (kBnd) {  // T's boundary values beside the stored nodes, corners included
                auto row_edges = [&](const E *Tr, int64_t b, bool whole) {
#pragma unroll
                    for (int i = 0; i < PX; ++i) {
                        if (!use[i]) continue;
                        const int gx = gx0 + 32 * i;
                        if (whole) T2[b + 32 * i] = Tr[32 * i];
                        if (gx == 1) T2[b + 32 * i - 1] = Tr[32 * i - 1];
                        if (gx == nx - 2) T2[b + 32 * i + 1] = Tr[32 * i + 1];
                    }
                };
                row_edges(Tc, base, false);
                if (gy == 1) row_edges(Tu, base - nx, true);
                if (gy == ny - 2) row_edges(Td, base + nx, true);
            }
        }
        if (!ok) {
            s_abort = 1;
            atomicOr(err, 1u);
        }
        __syncthreads();  // every thread is done with plane k's stage
        if (s_abort) {
            drain(min(k - 1 + NST, k1));
            return;
        }
        if (k + NST <= k1) issue(sk, k + NST);  // plane k's stage
        sk = sk1;
        dk = dk1;
#pragma unroll
        for (int i = 0; i < PX; ++i) {
            qm[i] = qc[i];
            qc[i] = qn[i];
        }
    }
}

}  // namespace psd
